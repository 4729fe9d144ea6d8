// kgs_sweep_dev.cuh -- device code shared by the sweep kernels: arithmetic
// helpers, the per-item partials and their ordered accumulator chains, and
// the persistent loop that claims work items.  Not part of the public ABI.
#pragma once

#include "kgs_internal.h"

namespace kgs {

// Raises the dynamic shared-memory limit of a kernel on the current device
// to at least `bytes`.
cudaError_t ensure_smem(const void *fn, size_t bytes);

namespace {

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 2^x - 1 with a relative error near FP32 rounding also for small x: for
// |x| < 1/4 the Taylor series of e^y - 1 in y = x ln 2 up to y^6 (the first
// omitted term is below 6e-9 of the sum), else the hardware 2^x minus 1
// (no cancellation beyond three bits there).
__device__ __forceinline__ float exp2m1(float x)
{
    const float y = x * 0.693147180559945309f;
    float p = fmaf(y, 1.f / 720.f, 1.f / 120.f);
    p = fmaf(p, y, 1.f / 24.f);
    p = fmaf(p, y, 1.f / 6.f);
    p = fmaf(p, y, 0.5f);
    const float small = fmaf(y * y, p, y);
    return fabsf(x) < 0.25f ? small : ex2_approx(x) - 1.f;
}

// exp of the scaled exponent: FP64 uses exp(), FP32 the hardware 2^x with the
// log2(e) factor already folded into the coefficient C_NEXP.
__device__ __forceinline__ double eq_exp(double x) { return exp(x); }
__device__ __forceinline__ float eq_exp(float x) { return ex2_approx(x); }
// FP64 implicit update: the reciprocal of the denominator from the hardware approximation
// refined by two Newton-Raphson steps r <- r + r (1 - den r) (quadratic
// convergence, about 1 ulp), then one product; den = 1/tau + sum a_d > 0.
__device__ __forceinline__ double implicit_div(double num, double den)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(den));
    r = fma(r, fma(-den, r, 1.0), r);
    r = fma(r, fma(-den, r, 1.0), r);
    return num * r;
}

__host__ __device__ constexpr size_t align16(size_t n) { return (n + 15) & ~size_t(15); }

// a - b = s + e exactly (Knuth's two-sum on a + (-b)).
template <typename Real>
__device__ __forceinline__ void two_diff(Real a, Real b, Real &s, Real &e)
{
    s = a - b;
    const Real bv = s - a;
    const Real av = s - bv;
    e = (a - av) - (b + bv);
}

// Running sum for the per-thread moment accumulation.  FP32 sums carry a
// Kahan compensation term (the value is sum - comp); FP64 sums are plain.
template <typename Real>
struct RunSum;
template <>
struct RunSum<float> {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        const float y = x - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};
template <>
struct RunSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ double value() const { return s; }
};

constexpr int VT = 8;  // moment-phase velocity table entries per velocity

// Four consecutive coefficients of a cell (one 16-byte shared load for FP32,
// two for FP64).
template <typename Real>
struct Quad {
    Real x, y, z, w;
};
__device__ __forceinline__ Quad<float> load_quad(const float *p)
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Quad<double> load_quad(const double *p)
{
    const double2 a = *reinterpret_cast<const double2 *>(p);
    const double2 b = *reinterpret_cast<const double2 *>(p + 2);
    return {a.x, a.y, b.x, b.y};
}
// Coefficient prefetch: each thread moves 8 of the slice's SLICE*NCOEF values.
constexpr int CPF = SLICE * NCOEF / NT;
static_assert(CPF == 8, "coefficient prefetch assumes 8 values per thread");
// Partial of one (group, cell) as stored in global memory: FP64, or the FP32
// Kahan pair (sum, compensation) with value sum - compensation.
template <typename Real>
struct PartOut;
template <>
struct PartOut<double> {
    using T = double;
};
template <>
struct PartOut<float> {
    using T = float2;
};

// (s0 - c0) + (s1 - c1) as a Kahan pair (s, c), value s - c, with an exact
// two-sum of the leading parts.
__device__ __forceinline__ float2 pair_add(float s0, float c0, float s1, float c1)
{
    const float S = s0 + s1;
    const float bv = S - s0;
    const float E = ((s0 - (S - bv)) + (s1 - bv)) - (c0 + c1);
    const float hi = S + E;
    const float lo = E - (hi - S);
    return make_float2(hi, -lo);
}

// Face-plane load: in the persistent kernel the value may have been written
// by another CTA during the same launch, so it bypasses L1 (the acquire of the
// upwind block's completion flag orders it after that CTA's stores).
template <bool COHERENT, typename Real>
__device__ __forceinline__ Real ld_face(const Real *p)
{
    if constexpr (COHERENT)
        return __ldcg(p);
    else
        return *p;
}
__device__ __forceinline__ int ld_acquire(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(int *p, int v)
{
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Bounded wait for a counter that only grows to reach `v`: its value then, or
// -1 after `limit` polls (the caller then records an error and returns).
__device__ inline int wait_count(const int *p, int v, long long limit)
{
    for (long long i = 0; i < limit; i++) {
        const int have = ld_acquire(p);
        if (have >= v) return have;
        __nanosleep(100);
    }
    return -1;
}

// Progress of a work item: the flag of (group, block) counts the slices whose
// x and y outflow is written, and becomes ITEM_DONE once the z outflow is
// too.  The block downwind in x or y sweeps its slice k as soon as slice k
// upwind is there, so neighbours overlap instead of running one after the
// other: with few items the time of an iteration is the longest chain of
// slices, (blocks along x + blocks along y - 2) * every + nz, instead of
// (stages) * bz.
constexpr int ITEM_DONE = 1 << 30;
// Lives in shared memory, used by thread 0 alone: in registers of every thread
// it would cost the sweep loop its last free ones.
struct Pipe {
    const int *up_x, *up_y;  // flags of the upwind blocks (null: none)
    int *own;                // this item's flag (null: never announced)
    int have;                // slices known to be there upwind
    int every;               // slices between announcements
    int go;                  // no wait of this item has expired
    long long limit;
    int *error;
    // Thread 0: wait until `need` slices are there upwind.  After an expired
    // wait the error word is set and the item runs on without waiting or
    // announcing (its results are discarded): an exit inside the slice loop
    // costs the loop's code about 10%.
    __device__ __forceinline__ void wait(int need)
    {
        if (have >= need) return;
        int n = ITEM_DONE;
        if (up_x) n = min(n, wait_count(up_x, need, limit));
        if (n > 0 && up_y) n = min(n, wait_count(up_y, need, limit));
        if (n < 0) {
            atomicExch(error, 1);
            go = 0;
            own = nullptr;
            n = ITEM_DONE;
        }
        have = n;
    }
    // Thread 0, after a barrier that follows the outflow stores of slice
    // done - 1 (the last slice is announced with the z outflow).  The barrier
    // and the release order every thread's stores before the flag.
    __device__ __forceinline__ void announce(int done, int of) const
    {
        if (own && done < of && done % every == 0) st_release(own, done);
    }
};

// Ordered accumulation of one item's moment partials.  Velocity group g (of
// all groups) adds into accumulator k = g % nacc; the items of one (k, block)
// form a chain in the order they were claimed, and the item at place `pos`
// adds after the one at pos - 1 (the first one stores).  The order is fixed
// by the work list, so the sums are bit-reproducible, and no item waits for
// one claimed after it.  FP32 partials are Kahan pairs (s, c) with value
// s - c; the accumulator holds a float-float pair (hi, lo) with value hi + lo,
// hi updated by a two-sum.
template <typename Real>
struct Acc16;
template <>
struct Acc16<double> {
    using V = double2;  // two slots
    __device__ static V init(V s) { return s; }
    __device__ static V add(V a, V s) { return make_double2(a.x + s.x, a.y + s.y); }
};
template <>
struct Acc16<float> {
    using V = float4;  // two slots: (s0, c0, s1, c1) / (hi0, lo0, hi1, lo1)
    __device__ static V init(V s) { return make_float4(s.x, -s.y, s.z, -s.w); }
    __device__ static float2 ff(float hi, float lo, float s, float c)
    {
        const float t = hi + s;
        const float bp = t - hi;
        const float err = (hi - (t - bp)) + (s - bp);
        return make_float2(t, lo + (err - c));
    }
    __device__ static V add(V a, V s)
    {
        const float2 p = ff(a.x, a.y, s.x, s.y), q = ff(a.z, a.w, s.z, s.w);
        return make_float4(p.x, p.y, q.x, q.y);
    }
};

// Block geometry of an item for the chain: physical extents and origin.
struct BlockSpan {
    bool px, py, pz;
    int x0, ex, y0, ey, z0, ez;
    __device__ BlockSpan(const SweepArgs &a, int o, int bxr, int byr, int bzr)
    {
        px = (o & 1) != 0, py = (o & 2) != 0, pz = (o & 4) != 0;
        const int bxi = px ? bxr : a.nbx - 1 - bxr;
        const int byi = py ? byr : a.nby - 1 - byr;
        const int bzi = pz ? bzr : a.nbz - 1 - bzr;
        x0 = bxi * BX, ex = min(BX, a.nx - x0);
        y0 = byi * BY, ey = min(BY, a.ny - y0);
        z0 = bzi * a.bz, ez = min(a.bz, a.nz - z0);
    }
    // global cell of the block's local (march-order) cell cl of slice lk
    __device__ size_t cell(const SweepArgs &a, int cl, int lk) const
    {
        const int li = cl % BX, lj = cl / BX;
        const int x = px ? x0 + li : x0 + ex - 1 - li;
        const int y = py ? y0 + lj : y0 + ey - 1 - lj;
        const int z = pz ? z0 + lk : z0 + ez - 1 - lk;
        return (size_t)x + (size_t)a.nx * ((size_t)y + (size_t)a.ny * z);
    }
    __device__ bool valid(int cl) const { return cl % BX < ex && cl / BX < ey; }
};

// Before the chain wait: pull the block's accumulator records into L2.
template <typename Real>
__device__ void chain_prefetch(const SweepArgs &a, const BlockSpan &b, int vgg)
{
    const unsigned char *acc = static_cast<const unsigned char *>(a.acc) +
                               (size_t)(vgg % a.nacc) * a.ncell * a.acc_slots * 8;
    const int rec = a.acc_slots * 8;
    for (int r = threadIdx.x; r < b.ez * BY; r += NT) {  // one row of ex cells
        const int lj = r % BY, lk = r / BY;
        if (lj >= b.ey) continue;
        const unsigned char *p = acc + b.cell(a, lj * BX, lk) * rec;
        const unsigned char *q = acc + b.cell(a, lj * BX + b.ex - 1, lk) * rec;
        const unsigned char *lo = p < q ? p : q;
        for (int off = 0; off < b.ex * rec; off += 128)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(lo + off));
    }
}

template <typename Real>
__device__ void chain_add(const SweepArgs &a, int o, int bxr, int byr, int bzr, int vgg, int pos,
                          const void *scratch)
{
    using Out = typename PartOut<Real>::T;
    const BlockSpan b(a, o, bxr, byr, bzr);
    const size_t ncell = a.ncell;
    if (a.acc_slots == ACC_COMPACT) {
        // the item's record and the accumulator record share one layout: add
        // them element-wise, 16 bytes (two slots) at a time, with CH vectors
        // of every thread in flight
        using A = Acc16<Real>;
        using V = typename A::V;
        constexpr int VPC = NPART * 8 / 16;  // vectors per cell record
        constexpr int CH = 4;
        const V *sc = static_cast<const V *>(scratch);
        V *acc = reinterpret_cast<V *>(static_cast<Out *>(a.acc) + (size_t)(vgg % a.nacc) * ncell * ACC_COMPACT);
        const int n = b.ez * SLICE * VPC;
        for (int base = threadIdx.x; base < n; base += NT * CH) {
            V sv[CH], av[CH];
            size_t at[CH];
            bool live[CH];
#pragma unroll
            for (int u = 0; u < CH; u++) {
                const int e = base + u * NT;
                const int lc = e / VPC, cl = lc % SLICE;
                live[u] = e < n && b.valid(cl);
                at[u] = live[u] ? b.cell(a, cl, lc / SLICE) * VPC + e % VPC : 0;
                if (live[u]) sv[u] = sc[e];  // written by this CTA: the same L1 path
            }
            if (pos > 0) {
#pragma unroll
                for (int u = 0; u < CH; u++)
                    if (live[u]) av[u] = __ldcg(acc + at[u]);
            }
#pragma unroll
            for (int u = 0; u < CH; u++)
                if (live[u]) acc[at[u]] = pos == 0 ? A::init(sv[u]) : A::add(av[u], sv[u]);
        }
        return;
    }
    // ACC_SPLIT: the item's flux slots go to the slots of the sides ahead of
    // its octant; the first item of the chain stores zero on the other sides
    const Out *sc = static_cast<const Out *>(scratch);
    Out *acc = static_cast<Out *>(a.acc) + (size_t)(vgg % a.nacc) * ncell * ACC_SPLIT;
    const int n = b.ez * SLICE * NPART;
#pragma unroll 4
    for (int e = threadIdx.x; e < n; e += NT) {
        const int q = e % NPART, cl = (e / NPART) % SLICE, lk = e / (NPART * SLICE);
        if (!b.valid(cl)) continue;
        const size_t cell = b.cell(a, cl, lk);
        const int slot = q < P_FX ? q : SUM_F0 + 2 * (q - P_FX) + ((o >> (q - P_FX)) & 1);
        const Out v = sc[e];  // written by this CTA: the same L1 path
        Out *dst = acc + cell * ACC_SPLIT + slot;
        if (pos == 0 && q >= P_FX) {
            Out *other = acc + cell * ACC_SPLIT + (SUM_F0 + 2 * (q - P_FX) + 1 - ((o >> (q - P_FX)) & 1));
            if constexpr (sizeof(Real) == 8)
                *other = 0.0;
            else
                *other = make_float2(0.f, 0.f);
        }
        if constexpr (sizeof(Real) == 8) {
            *dst = pos == 0 ? v : __ldcg(dst) + v;
        } else {
            if (pos == 0) {
                *dst = make_float2(v.x, -v.y);
            } else {
                const float2 cur = __ldcg(dst);
                const float t = cur.x + v.x;
                const float bp = t - cur.x;
                const float err = (cur.x - (t - bp)) + (v.x - bp);
                *dst = make_float2(t, cur.y + (err - v.y));
            }
        }
    }
}
// Persistent sweep over the items of many problem instances.  Items are
// claimed in list order (stage-major), so every item's upwind dependencies
// and its accumulator-chain predecessor were claimed earlier by CTAs that are
// running: the waits always end unless an error stopped a producer, and then
// they end at the poll limit.
template <typename Real, typename Item>
__device__ __forceinline__ void persistent_loop(const BatchSweepArgs &b, Item item_sweep)
{
    __shared__ SweepArgs sa;
    __shared__ Pipe pipe;
    __shared__ int s_item, s_go;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(b.counter, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= b.n_items) break;
        const int4 item = b.items[it];
        const int inst = item.x, o = item.y >> 24, vg = item.y & 0xffffff;
        const int bxr = item.z & 1023, byr = (item.z >> 10) & 1023, bzr = (item.z >> 20) & 1023;
        // copy the instance's arguments to shared memory (words of the struct)
        {
            const int *src = reinterpret_cast<const int *>(b.inst + inst);
            int *dst = reinterpret_cast<int *>(&sa);
            for (int q = threadIdx.x; q < (int)(sizeof(SweepArgs) / sizeof(int)); q += NT) dst[q] = src[q];
        }
        if (threadIdx.x == 0) {
            const SweepArgs &a = b.inst[inst];
            const int vgg = item.w;  // global velocity-group index within the instance
            int *own = b.flags + b.flag_off[inst] + ((vgg * a.nbz + bzr) * a.nby + byr) * a.nbx + bxr;
            pipe.up_x = bxr > 0 ? own - 1 : nullptr;
            pipe.up_y = byr > 0 ? own - a.nbx : nullptr;
            pipe.own = it != b.skip_publish ? own : nullptr;
            pipe.have = 0;
            pipe.every = b.announce_every;
            pipe.limit = b.spin_limit;
            pipe.error = b.error;
            bool ok = *b.error == 0;
            if (ok && bzr > 0) {
                ok = wait_count(own - a.nbx * a.nby, ITEM_DONE, b.spin_limit) >= 0;
                if (!ok) atomicExch(b.error, 1);
            }
            pipe.go = ok;
            if (ok) pipe.wait(1);
            s_go = pipe.go;
        }
        __syncthreads();
        // not pipe.go: thread 0 may be in the item already and clear it there
        if (!s_go) break;
        void *scratch = static_cast<unsigned char *>(b.scratch) + (size_t)blockIdx.x * b.scratch_stride;
        item_sweep(sa, make_int4(o, bxr, byr, bzr), vg, scratch, pipe);
        __syncthreads();
        if (!pipe.go) break;
        // the downwind blocks may finish: the face planes are written
        if (threadIdx.x == 0 && pipe.own) st_release(pipe.own, ITEM_DONE);
        // then the item's turn in its accumulator chain
        const int pos = b.pos[it], vgg = item.w;
        const int bxi = (o & 1) ? bxr : sa.nbx - 1 - bxr;
        const int byi = (o & 2) ? byr : sa.nby - 1 - byr;
        const int bzi = (o & 4) ? bzr : sa.nbz - 1 - bzr;
        int *tk = sa.tok + (((size_t)(vgg % sa.nacc) * sa.nbz + bzi) * sa.nby + byi) * sa.nbx + bxi;
        if (pos > 0) chain_prefetch<Real>(sa, BlockSpan(sa, o, bxr, byr, bzr), vgg);
        if (threadIdx.x == 0) {
            bool ok = pos == 0 || wait_count(tk, pos, b.spin_limit) >= 0;
            if (!ok) atomicExch(b.error, 1);
            s_go = ok ? 1 : 0;
        }
        __syncthreads();
        if (!s_go) break;
        chain_add<Real>(sa, o, bxr, byr, bzr, vgg, pos, scratch);
        __syncthreads();
        if (threadIdx.x == 0) st_release(tk, pos + 1);
    }
}

}  // namespace
}  // namespace kgs
