// kgs_sweep_f2.cu -- the FP32 sweep with two neighbouring velocities per
// thread and packed FP32 arithmetic (arXiv 1810.00348, Eqs. (2), (5), (7),
// (9)).  The work decomposition is that of kgs_sweep.cu; what differs is how
// a thread block works through its item.
//
// What bounds it.  A block holds one slice of 256 velocities in shared memory
// (83 KB, 87.5 KB with its tables), so two blocks of four warps share an SM and the kernel is
// bound by the issue slots of two warps per scheduler and by the latency of
// their dependent chains, not by a pipe or by memory.  The packed forms
// (fma.rn.f32x2 and its kin: two FP32 results per lane and instruction, each
// rounded as the scalar instruction rounds it) run at half the issue rate of
// the scalar ones with the same latency, so they leave the arithmetic rate
// unchanged and halve the issue slots (measured per SM and clock: 1.73 packed
// against 3.86 scalar FMAs, 4.8 cycles from one to the next that needs it).
// To use them without moves the two velocities of a thread sit in neighbouring slots (2t
// and 2t + 1 of its group), which the host orders (pack_order) so that they
// have the same x node on neighbouring x-lines: face planes and slice
// positions move as 8-byte words, and the moment phase sums two lines at
// once, each in its own half and in node order, so that every sum keeps the
// order it has with one line at a time.
//
// Layout of the slice: the 64 cells of the block with a pitch of 8, then the
// 8 cells of the halo column and the 8 of the halo row; the stride of a cell,
// 129 8-byte words, is odd, so that the moment phase (a cell per lane) reads
// without bank conflicts.
//
// Measured against the same work with one scalar chain per velocity: 39.8
// instead of 54.7 instructions per phase point; 64^3 cells x 32^3 velocities
// 24.3 -> 20.4 ms (19.1 with the diagonals stored once computed), 96x64x64 x
// 48^3 with a solid cube 146 -> 111 ms, growing cells (50x43x43 x 24^3) 8.06 ->
// 5.84 ms.  The results are the same bit for bit: every sum keeps its order,
// and the only products that are not rounded by themselves are those that
// enter a compensated sum alone.
#include "kgs_pack.h"
#include "kgs_sweep_dev.cuh"

namespace kgs {
namespace {

constexpr int VG = 2 * NT;       // velocity slots per group, at most
constexpr int CSP = VG / 2 + 1;  // 8-byte words per cell of the slice
constexpr int HCOL = SLICE, HROW = SLICE + BY, NPOS = SLICE + BY + BX;
constexpr int LREC = 8;          // floats of a row of SweepArgs::lines
static_assert(sizeof(float2) * BX * CSP >= sizeof(float2) * NPART * SLICE, "reduction buffer in the halo row");

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a - b (exactly the rounding of a subtraction: the product by -1 is exact)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// Two running Kahan sums (value s + n: n is the negated compensation).
struct KahanPair {
    float2 s = make_float2(0.f, 0.f), n = make_float2(0.f, 0.f);
    __device__ __forceinline__ void add(float2 x)
    {
        const float2 y = add2(x, n);
        const float2 t = add2(s, y);
        n = add2(y, sub2(s, t));
        s = t;
    }
    // add a * b, the product not rounded by itself
    __device__ __forceinline__ void add_mul(float2 a, float2 b)
    {
        const float2 y = fma2(a, b, n);
        const float2 t = add2(s, y);
        n = add2(y, sub2(s, t));
        s = t;
    }
};

// Sums over the x nodes of two lines, one in each half: P_a = sum w_x c_x^a g,
// C_a = the first-order correction of P_a for the low part of c_x.
struct LineSums {
    float2 P0 = make_float2(0.f, 0.f), P1 = P0, P2 = P0, P3 = P0, C1 = P0, C2 = P0, C3 = P0;
    __device__ __forceinline__ void add(float2 f, float2 w, float2 h, float2 l)
    {
        const float2 t0 = mul2(w, f);
        const float2 t1 = mul2(t0, h);
        const float2 t2 = mul2(t1, h);
        P0 = add2(P0, t0);
        P1 = add2(P1, t1);
        P2 = add2(P2, t2);
        P3 = fma2(t2, h, P3);
        C1 = fma2(t0, l, C1);
        C2 = fma2(t1, l, C2);
        C3 = fma2(t2, l, C3);
    }
};

struct Layout2 {
    static constexpr size_t off_coef = align16(sizeof(float2) * NPOS * CSP);
    static constexpr size_t off_x = off_coef + sizeof(float) * SLICE * NCOEF;
    // x nodes of the octant (xi_x, its low part, w_x, -)
    __host__ __device__ static size_t off_cx(int nxm) { return off_x + sizeof(float4) * nxm; }
    // c_x tables of lines that do not have 16 nodes: [2][SLICE][cxs], an odd stride
    __host__ __device__ static int cxs(int nxm) { return nxm | 1; }
    __host__ __device__ static size_t off_line(int nxm, bool line16)
    {
        return off_cx(nxm) + (line16 ? 0 : align16(2 * sizeof(float) * SLICE * cxs(nxm)));
    }
    static size_t total(int nxm, bool line16, int lines_max)
    {
        return off_line(nxm, line16) + sizeof(float) * LREC * lines_max;
    }
};

// Barrier of the two warps that sum the two halves of the same 32 cells.
__device__ __forceinline__ void pair_barrier()
{
    asm volatile("bar.sync %0, 64;" ::"r"(1 + (int)(threadIdx.x / 32) % 2) : "memory");
}

// One work item (see sweep_item of kgs_sweep.cu for the meaning of the
// arguments and of the partials that it writes).
//   LINE   16: every x-line has 16 slots, whose c_x stay in registers
//   UNIF   equal cell widths along each axis
//   DEV    the deviation-form source (uniform grids)
template <int LINE, bool COHERENT, bool UNIF, bool DEV>
__device__ __forceinline__ void sweep_item2(const SweepArgs &a, const int4 w, const int vgy, unsigned char *smem,
                                            void *scratch, Pipe *pipe)
{
    static_assert(!DEV || UNIF, "the deviation-form source needs a uniform grid");
    const int nxm = a.nxo_max;
    float2 *slice = reinterpret_cast<float2 *>(smem);
    float *cs = reinterpret_cast<float *>(smem + Layout2::off_coef);
    float4 *xn = reinterpret_cast<float4 *>(smem + Layout2::off_x);
    const int cxs = Layout2::cxs(nxm);
    float *cxh = reinterpret_cast<float *>(smem + Layout2::off_cx(nxm));  // [SLICE][cxs]
    float *cxl = cxh + SLICE * cxs;
    float *lrec = reinterpret_cast<float *>(smem + Layout2::off_line(nxm, LINE > 0));
    float2 *red = slice + HROW * CSP;  // [NPART][SLICE]: the halo row is not read during the moment phase

    const int t = threadIdx.x;
    const int o = w.x;
    const int vcount = a.oct_vcount[o];
    const int v0 = vgy * VG;
    if (v0 >= vcount) return;
    const int nvg = min(VG, vcount - v0);
    const int gvbase = a.oct_vstart[o] + v0;
    const int vgid = a.oct_vgbase[o] + vgy;
    const int nxo = a.oct_nx[o];
    const int line0 = v0 / nxo;  // first line of the octant that the group touches

    const bool px = (o & 1) != 0, py = (o & 2) != 0, pz = (o & 4) != 0;
    const int bxi = px ? w.y : a.nbx - 1 - w.y;
    const int byi = py ? w.z : a.nby - 1 - w.z;
    const int bzi = pz ? w.w : a.nbz - 1 - w.w;
    const int x0 = bxi * BX, ex = min(BX, a.nx - x0);
    const int y0 = byi * BY, ey = min(BY, a.ny - y0);
    const int z0 = bzi * a.bz, ez = min(a.bz, a.nz - z0);
    const bool xfirst = w.y == 0, yfirst = w.z == 0, zfirst = w.w == 0;
    const bool xlast = w.y == a.nbx - 1, ylast = w.z == a.nby - 1, zlast = w.w == a.nbz - 1;
    const int sidex = px ? 0 : 1, sidey = py ? 2 : 3, sidez = pz ? 4 : 5;  // upwind sides
    const int headx = px ? 1 : 0, heady = py ? 3 : 2, headz = pz ? 5 : 4;  // downwind sides
    const int nx = a.nx, ny = a.ny;
    const size_t ncell = a.ncell;
    const size_t Nv = (size_t)a.Nv;
    const bool any_solid =
        a.any_solid != 0 && !(a.blk_plain != nullptr && a.blk_plain[((size_t)bzi * a.nby + byi) * a.nbx + bxi] != 0);
    // The unrolled diagonals sweep all 64 cells of a block without solid
    // cells; the cells past a ragged edge take part (nothing flows from them
    // into the block, and the moments skip them) while that is less work than
    // the loop over the diagonals that are there, which costs about 1.5 times
    // as much per cell.
    const bool unrolled = !any_solid && 3 * ex * ey >= 2 * SLICE;

    auto GX = [&](int li) { return px ? x0 + li : x0 + ex - 1 - li; };
    auto GY = [&](int lj) { return py ? y0 + lj : y0 + ey - 1 - lj; };
    auto GZ = [&](int lk) { return pz ? z0 + lk : z0 + ez - 1 - lk; };
    auto POS = [](int li, int lj) { return lj < 0 ? HROW + li : li < 0 ? HCOL + lj : lj * BX + li; };
    auto CELL = [&](int x, int y, int z) { return (size_t)x + (size_t)nx * ((size_t)y + (size_t)ny * z); };

    const float *vel = static_cast<const float *>(a.vel);
    const float *velm = static_cast<const float *>(a.velm);
    const float *mt = static_cast<const float *>(a.mtab);
    const float *coef = static_cast<const float *>(a.coef);
    float *FXp = static_cast<float *>(a.FX);
    float *FYp = static_cast<float *>(a.FY);
    float *FZp = static_cast<float *>(a.FZ);

    // ---- the thread's two velocities and the moment-phase tables ----
    // The sweep carries g = f - M_ref; ghosts enter as ghost - M_ref.
    const bool ok = 2 * t < nvg;
    const size_t gv = (size_t)gvbase + (ok ? 2 * t : 0);
    float2 xi[3], axi[3], adx[3], asum = f2(0.f), xsq, mref, dmref = f2(0.f);
    {
        const float4 p = *reinterpret_cast<const float4 *>(vel + gv * 4);
        const float4 q = *reinterpret_cast<const float4 *>(vel + gv * 4 + 4);
        xi[0] = make_float2(p.x, q.x);
        xi[1] = make_float2(p.y, q.y);
        xi[2] = make_float2(p.z, q.z);
        xsq = make_float2(velm[gv * 8 + 7], velm[gv * 8 + 15]);
        mref = make_float2(velm[gv * 8 + 5], velm[gv * 8 + 13]);
        if constexpr (DEV) dmref = make_float2(velm[gv * 8 + 6], velm[gv * 8 + 14]);
    }
#pragma unroll
    for (int d = 0; d < 3; d++) {
        axi[d] = make_float2(fabsf(xi[d].x), fabsf(xi[d].y));
        adx[d] = UNIF ? mul2(axi[d], f2((float)a.rd0[d])) : f2(0.f);
    }
    if constexpr (UNIF) asum = add2(add2(adx[0], adx[1]), adx[2]);
    const float2 nmref = make_float2(-mref.x, -mref.y);
    auto row2 = [&](int row) { return *reinterpret_cast<const float2 *>(mt + (size_t)row * Nv + gv); };
    const float2 mgx = row2(a.side_inflow[sidex] ? MT_INFLOW : sidex);
    const float2 mgy = row2(a.side_inflow[sidey] ? MT_INFLOW : sidey);
    // ghost value rho_w * (unit wall or free-stream Maxwellian) - M_ref
    auto ghost = [&](float rw, float2 mg) { return fma2(f2(rw), mg, nmref); };
    {
        const int nlines = (v0 + nvg - 1) / nxo - line0 + 1;
        const float4 *src = reinterpret_cast<const float4 *>(a.lines + ((size_t)a.oct_line0[o] + line0) * LREC);
        for (int l = t; l < 2 * nlines; l += NT) reinterpret_cast<float4 *>(lrec)[l] = src[l];
        const float4 *xs = reinterpret_cast<const float4 *>(a.xnodes) + (size_t)o * a.xn_stride;
        for (int ix = t; ix < nxo; ix += NT) xn[ix] = xs[ix];
    }
    // the half of the group that this thread sums in the moment phase
    static_assert(PACK_HALF == NT, "a thread sums one half of the group");
    const int mcl = t % SLICE, mvp = t / SLICE;  // NT = 2 * SLICE
    const int mb = mvp * NT, mn = min(NT, nvg - mb);
    const PackHalf half(v0 + mb, mn, nxo);
    const int head = half.head, full = half.full, tail = half.tail;
    const int first = LINE > 0 ? nxo - head : half.first;  // node of the head's first velocity (16: no line is cut)
    const int mline = mn > 0 ? (v0 + mb) / nxo - line0 : 0;  // line of its first velocity

    // the persistent sweep reads the wall densities in FP32: converting them
    // here would take a 64-cycle FP64-pipe instruction per value and warp
    auto rho_wall = [&](int side, size_t cell) -> float {
        return COHERENT ? a.rho_w32[side * ncell + cell] : (float)a.rho_w[side * ncell + cell];
    };
    auto wall_rho = [&](int side, size_t cell) -> float {
        return a.side_inflow[side] ? 1.f : rho_wall(side, cell);
    };
    auto ld2 = [](const float *p) { return ld_face<COHERENT>(reinterpret_cast<const float2 *>(p)); };

    // ---- prefetch registers: coefficients and halos of one slice ----
    float pc[CPF];
    float2 phx[BY], phy[BX];
    auto prefetch = [&](int lk) {
        const int z = GZ(lk);
        const int cl = (t * CPF) / NCOEF, q0 = (t * CPF) % NCOEF;
        const int li = cl % BX, lj = cl / BX;
        if (li < ex && lj < ey) {
            const float4 *src = reinterpret_cast<const float4 *>(coef + CELL(GX(li), GY(lj), z) * NCOEF + q0);
            const float4 c0 = src[0], c1 = src[1];
            pc[0] = c0.x, pc[1] = c0.y, pc[2] = c0.z, pc[3] = c0.w;
            pc[4] = c1.x, pc[5] = c1.y, pc[6] = c1.z, pc[7] = c1.w;
        } else {
#pragma unroll
            for (int q = 0; q < CPF; q++) pc[q] = (q0 + q == C_FLAGS) ? flag_value<float>(F_SOLID) : 0.f;
        }
        if (xfirst) {
#pragma unroll
            for (int lj2 = 0; lj2 < BY; lj2++) {
                if (lj2 >= ey) break;
                phx[lj2] = ghost(wall_rho(sidex, CELL(GX(0), GY(lj2), z)), mgx);
            }
        } else {
            const float *fi = FXp + ((size_t)z * ny + GY(0)) * Nv + gv;
            const long long step = py ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int lj2 = 0; lj2 < BY; lj2++) {
                if (lj2 >= ey) break;
                phx[lj2] = ld2(fi + lj2 * step);
            }
        }
        if (yfirst) {
#pragma unroll
            for (int li2 = 0; li2 < BX; li2++) {
                if (li2 >= ex) break;
                phy[li2] = ghost(wall_rho(sidey, CELL(GX(li2), GY(0), z)), mgy);
            }
        } else {
            const float *fi = FYp + ((size_t)z * nx + GX(0)) * Nv + gv;
            const long long step = px ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int li2 = 0; li2 < BX; li2++) {
                if (li2 >= ex) break;
                phy[li2] = ld2(fi + li2 * step);
            }
        }
    };
    prefetch(0);

    // z inflow of the block: the slice starts as slice k0 - 1.  A row of cells
    // is loaded before it is stored, so a row's loads are in flight together.
    if (zfirst) {
        const float2 mgz = row2(a.side_inflow[sidez] ? MT_INFLOW : sidez);
        for (int lj = 0; lj < ey; lj++)
            for (int li = 0; li < ex; li++) {
                const float rw = wall_rho(sidez, CELL(GX(li), GY(lj), GZ(0)));
                if (ok) slice[(lj * BX + li) * CSP + t] = ghost(rw, mgz);
            }
    } else {
        const long long sx = px ? (long long)Nv : -(long long)Nv;
        for (int lj = 0; lj < ey; lj++) {
            const float *fi = FZp + ((size_t)GY(lj) * nx + GX(0)) * Nv + gv;
            float2 v[BX];
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
                v[li] = ld2(fi + li * sx);
            }
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
                if (ok) slice[(lj * BX + li) * CSP + t] = v[li];
            }
        }
    }

    for (int lk = 0; lk < ez; lk++) {
        const int z = GZ(lk);
        // stage the prefetched slice data in shared memory
#pragma unroll
        for (int q = 0; q < CPF; q += 4)
            *reinterpret_cast<float4 *>(cs + t * CPF + q) = make_float4(pc[q], pc[q + 1], pc[q + 2], pc[q + 3]);
        if (ok) {
#pragma unroll
            for (int lj = 0; lj < BY; lj++) slice[(HCOL + lj) * CSP + t] = phx[lj];
#pragma unroll
            for (int li = 0; li < BX; li++) slice[(HROW + li) * CSP + t] = phy[li];
        }
        if (COHERENT && t == 0) pipe->wait(min(lk + 2, ez));
        __syncthreads();
        // c_x = xi_x - U_x of each cell of the slice as a float pair, per x slot
        if constexpr (LINE == 0) {
            const float ux = -0.5f * cs[mcl * NCOEF + C_M2UX];
            for (int ix = mvp; ix < nxo; ix += NT / SLICE) {
                float s, e;
                two_diff(xn[ix].x, ux, s, e);
                cxh[mcl * cxs + ix] = s;
                cxl[mcl * cxs + ix] = e + xn[ix].y;
            }
        }
        if (lk + 1 < ez) prefetch(lk + 1);

        // ---- sweep of the slice: Eq. (2) fused into Eq. (7), by anti-diagonals ----
        // The update is written about the upwind x value,
        //   f = f_x + (src - f_x/tau + a_y (f_y - f_x) + a_z (f_z - f_x)) / den:
        // on a smooth field the increment is small and the one rounding that
        // matters is the final, unbiased addition.
        auto cell_update = [&](const float *c, float2 fx, float2 fy, float2 fz) -> float2 {
            const Quad<float> c0 = load_quad(c), c1 = load_quad(c + 4), c2 = load_quad(c + 8), c3 = load_quad(c + 12);
            const float2 cq = fma2(xi[0], f2(c2.x), fma2(xi[1], f2(c2.y), fma2(xi[2], f2(c2.z), f2(c3.w))));
            const float2 nrtau = f2(-c1.z);
            if constexpr (DEV) {
                // rtau (f^S - M_ref) as rtau M_ref (2^D shak - 1), D = log2(f^S_M / M_ref)
                // from terms that vanish at the reference state
                const float2 sd = fma2(xi[0], f2(c0.x), fma2(xi[1], f2(c0.y), mul2(xi[2], f2(c0.z))));
                const float2 D = fma2(xsq, f2(c2.w), fma2(sd, f2(c1.x), f2(c3.x)));
                const float2 shm1 = mul2(cq, fma2(add2(xsq, sd), f2(c1.y), f2(c3.z)));
                // 2^D - 1: the series of e^y - 1 below 1/4, the hardware 2^x beyond
                const float2 y = mul2(D, f2(0.693147180559945309f));
                float2 p = fma2(y, f2(1.f / 720.f), f2(1.f / 120.f));
                p = fma2(p, y, f2(1.f / 24.f));
                p = fma2(p, y, f2(1.f / 6.f));
                p = fma2(p, y, f2(0.5f));
                float2 em = fma2(mul2(y, y), p, y);
                if (!(fabsf(D.x) < 0.25f)) em.x = ex2_approx(D.x) - 1.f;
                if (!(fabsf(D.y) < 0.25f)) em.y = ex2_approx(D.y) - 1.f;
                const float2 X = fma2(em, shm1, add2(em, shm1));
                const float2 dsrc = mul2(f2(c1.z), fma2(mref, X, dmref));
                float2 r = fma2(nrtau, fx, dsrc);
                r = fma2(adx[1], sub2(fy, fx), r);
                r = fma2(adx[2], sub2(fz, fx), r);
                const float2 den = add2(f2(c1.z), asum);
                return fma2(r, make_float2(rcp_approx(den.x), rcp_approx(den.y)), fx);
            } else {
                // |c|^2 - |U|^2 = |xi|^2 - 2 U.xi and c.q' = xi.q' - U.q'
                const float2 s = fma2(xi[0], f2(c0.x), fma2(xi[1], f2(c0.y), fma2(xi[2], f2(c0.z), xsq)));
                const float2 shak = fma2(cq, fma2(s, f2(c1.y), f2(c3.z)), f2(1.f));
                const float2 ar = fma2(s, f2(c1.x), f2(c0.w));
                const float2 src = mul2(make_float2(ex2_approx(ar.x), ex2_approx(ar.y)), shak);
                float2 ay, az, den;
                if constexpr (UNIF) {
                    ay = adx[1];
                    az = adx[2];
                    den = add2(f2(c1.z), asum);
                } else {
                    ay = mul2(axi[1], f2(c3.x));
                    az = mul2(axi[2], f2(c3.y));
                    den = add2(add2(fma2(axi[0], f2(c2.w), f2(c1.z)), ay), az);
                }
                float2 r = fma2(nrtau, add2(fx, mref), src);
                r = fma2(ay, sub2(fy, fx), r);
                r = fma2(az, sub2(fz, fx), r);
                return fma2(r, make_float2(rcp_approx(den.x), rcp_approx(den.y)), fx);
            }
        };
        if (unrolled) {
            // The 15 diagonals unrolled: the upwind x and y values of a cell
            // were computed on the previous diagonal by this thread and stay
            // in registers (prev[row]); the z value (the cell itself in slice
            // k - 1) and the halo come from shared memory.  A diagonal is
            // stored once all its cells are computed: a store between them
            // would keep the compiler from moving the next cell's shared
            // loads above it (64^3 x 32^3: 19.7 -> 19.3 ms, cube 116 -> 113).
            float2 prev[BY];
#pragma unroll
            for (int d = 0; d < BX + BY - 1; d++) {
#pragma unroll
                for (int k = 0; k < BY; k++) {
                    const int lj = (d < BY - 1 ? d : BY - 1) - k;
                    const int li = d - lj;
                    if (lj >= 0 && li < BX) {
                        const float2 fz = slice[(lj * BX + li) * CSP + t];
                        const float2 fx = li == 0 ? slice[(HCOL + lj) * CSP + t] : prev[lj];
                        const float2 fy = lj == 0 ? slice[(HROW + li) * CSP + t] : prev[lj > 0 ? lj - 1 : 0];
                        const float2 f = cell_update(cs + (lj * BX + li) * NCOEF, fx, fy, fz);
                        prev[lj] = f;
                    }
                }
                if (ok) {
#pragma unroll
                    for (int k = 0; k < BY; k++) {
                        const int lj = (d < BY - 1 ? d : BY - 1) - k, li = d - lj;
                        if (lj >= 0 && li < BX) slice[(lj * BX + li) * CSP + t] = prev[lj];
                    }
                }
            }
        } else {
            // The upwind values of cell (i, j) are read from the in-place
            // slice: (i-1, j) and (i, j-1) were updated on the previous
            // diagonal, (i, j) itself still holds slice k - 1.
            for (int d = 0; d < ex + ey - 1; d++) {
                const int jhi = min(ey - 1, d), jlo = max(0, d - (ex - 1));
#pragma unroll
                for (int k = 0; k < BY; k++) {
                    const int lj = jhi - k;
                    if (lj >= jlo) {
                        const int li = d - lj;
                        const float *c = cs + (lj * BX + li) * NCOEF;
                        const int flags = any_solid ? flag_bits(c[C_FLAGS]) : 0;
                        if (!(flags & F_SOLID)) {
                            float2 *at = slice + (lj * BX + li) * CSP + t;
                            float2 fz = *at;
                            float2 fy = slice[POS(li, lj - 1) * CSP + t];
                            float2 fx = slice[POS(li - 1, lj) * CSP + t];
                            if (flags) {
                                const size_t cell = CELL(GX(li), GY(lj), z);
                                const float2 msol = row2(MT_SOLID);
                                if (flags & (F_SOLID_SIDE << sidex))
                                    fx = ghost(rho_wall(sidex, cell), msol);
                                if (flags & (F_SOLID_SIDE << sidey))
                                    fy = ghost(rho_wall(sidey, cell), msol);
                                if (flags & (F_SOLID_SIDE << sidez))
                                    fz = ghost(rho_wall(sidez, cell), msol);
                            }
                            const float2 f = cell_update(c, fx, fy, fz);
                            if (ok) *at = f;
                        }
                    }
                }
            }
        }
        // outflow of the slice through the block's downwind x and y faces
        // (own velocities, read back from the slice)
        if (!xlast && ok) {
            float *fo = FXp + ((size_t)z * ny + GY(0)) * Nv + gv;
            const long long step = py ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int lj = 0; lj < BY; lj++) {
                if (lj >= ey) break;
                *reinterpret_cast<float2 *>(fo + lj * step) = slice[(lj * BX + ex - 1) * CSP + t];
            }
        }
        if (!ylast && ok) {
            float *fo = FYp + ((size_t)z * nx + GX(0)) * Nv + gv;
            const long long step = px ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
                *reinterpret_cast<float2 *>(fo + li * step) = slice[((ey - 1) * BX + li) * CSP + t];
            }
        }
        // the moment phase's cell: read before the barrier that frees the staged record
        const float *mc = cs + mcl * NCOEF;
        const int mflags = flag_bits(mc[C_FLAGS]);
        const float ux = -0.5f * mc[C_M2UX];
        const float2 uyz = make_float2(-0.5f * mc[C_M2UY], -0.5f * mc[C_M2UZ]);
        __syncthreads();
        if (COHERENT && t == 0) pipe->announce(lk + 1, ez);

        // ---- moments of the slice over the group's velocities ----
        {
            const int cl = mcl, vp = mvp;
            const int li = cl % BX, lj = cl / BX;
            const bool valid = li < ex && lj < ey;
            const int flags = mflags;
            // running sums in pairs of slots: (S0, S1x) (S1y, S1z) (S2yy, S2zz)
            // (S2xy, S2xz) (S2xx, S2yz) (S3y, S3z) (S3x, Fx) (Fy, Fz)
            KahanPair S[8];
            if (valid && !(flags & F_SOLID)) {
                const bool wx = flags & (F_WALL_SIDE << headx);
                const bool wy = flags & (F_WALL_SIDE << heady);
                const bool wz = flags & (F_WALL_SIDE << headz);
                const float sgnx = px ? 1.f : -1.f;
                // fold the sums P_a of line l with its c_y, c_z and w_y w_z
                auto fold = [&](float P0, float P1, float P2, float P3, int l) {
                    const float4 e = *reinterpret_cast<const float4 *>(lrec + l * LREC);
                    const float2 v = make_float2(e.x, e.y);
                    // two-difference: v - u = cc + its error
                    const float2 cc = sub2(v, uyz);
                    const float2 bv = sub2(cc, v);
                    const float2 av = sub2(cc, bv);
                    const float2 cl2 =
                        add2(sub2(sub2(v, av), add2(uyz, bv)), make_float2(e.w, lrec[l * LREC + 4]));
                    const float W = e.z;
                    const float2 q01 = mul2(f2(W), make_float2(P0, P1));
                    const float q0 = q01.x, q1 = q01.y, q2 = W * P2;
                    S[0].add(q01);
                    S[1].add(fma2(cc, f2(q0), mul2(cl2, f2(q0))));
                    const float2 ccl = mul2(cc, cl2);
                    S[2].add_mul(fma2(cc, cc, add2(ccl, ccl)), f2(q0));
                    S[3].add(fma2(cc, f2(q1), mul2(cl2, f2(q1))));
                    const float yz = fmaf(cc.x, cc.y, fmaf(cl2.x, cc.y, cc.x * cl2.y));
                    S[4].add_mul(make_float2(1.f, yz), make_float2(q2, q0));
                    const float r2 = fmaf(cc.x, cc.x, cc.y * cc.y);
                    const float r2l = 2.f * fmaf(cc.x, cl2.x, cc.y * cl2.y);
                    const float e2 = fmaf(r2, q0, fmaf(r2l, q0, q2));
                    S[5].add(fma2(cc, f2(e2), mul2(cl2, f2(e2))));
                    // incoming flux w |xi_d| f towards the wall ahead
                    S[6].add(make_float2(fmaf(W, P3, fmaf(r2, q1, r2l * q1)), wx ? sgnx * fmaf(ux, q0, q1) : 0.f));
                    if (wy || wz)
                        S[7].add_mul(make_float2(fabsf(v.x), fabsf(v.y)), make_float2(wy ? q0 : 0.f, wz ? q0 : 0.f));
                };
                float hr[LINE > 0 ? LINE : 1], lr[LINE > 0 ? LINE : 1];
                if constexpr (LINE > 0) {
#pragma unroll
                    for (int ix = 0; ix < LINE; ix++) {
                        const float4 n = xn[ix];
                        float e;
                        two_diff(n.x, ux, hr[ix], e);
                        lr[ix] = e + n.y;
                    }
                }
                const float *hc = cxh + cl * cxs, *lc = cxl + cl * cxs;
                const float2 *sp = slice + cl * CSP + mb / 2;
                // the units of the half in line order (PackHalf)
                const int pairs = full / 2;
                const int n_units = (head > 0) + pairs + (full & 1) + (tail > 0);
                const float *seq = reinterpret_cast<const float *>(sp + pairs * nxo);  // the unpaired ones
                int line = mline;
                for (int u = 0; u < n_units; u++) {
                    const int k = u - (head > 0);
                    const bool two = k >= 0 && k < pairs;
                    LineSums P;
                    if (two) {
                        const float2 *fl = sp + k * nxo;
                        if constexpr (LINE > 0) {
#pragma unroll
                            for (int ix = 0; ix < LINE; ix++) P.add(fl[ix], f2(xn[ix].z), f2(hr[ix]), f2(lr[ix]));
                        } else {
#pragma unroll 4
                            for (int ix = 0; ix < nxo; ix++) P.add(fl[ix], f2(xn[ix].z), f2(hc[ix]), f2(lc[ix]));
                        }
                    } else {
                        const int n = k < 0 ? head : (k == pairs && (full & 1)) ? nxo : tail;
                        const int ix0 = k < 0 ? first : 0;
                        for (int ix = ix0; ix < ix0 + n; ix++) {
                            float hi, lo;
                            if constexpr (LINE > 0) {
                                float e;
                                two_diff(xn[ix].x, ux, hi, e);
                                lo = e + xn[ix].y;
                            } else {
                                hi = hc[ix];
                                lo = lc[ix];
                            }
                            P.add(f2(*seq++), f2(xn[ix].z), f2(hi), f2(lo));
                        }
                    }
                    // first-order corrections for the low part of c_x
                    const float2 P1 = add2(P.P1, P.C1), P2 = fma2(f2(2.f), P.C2, P.P2), P3 = fma2(f2(3.f), P.C3, P.P3);
#pragma unroll 1
                    for (int h = 0; h <= (int)two; h++)
                        fold(h ? P.P0.y : P.P0.x, h ? P1.y : P1.x, h ? P2.y : P2.x, h ? P3.y : P3.x, line++);
                }
            }
            // combine the two halves and write the (group, cell) partial:
            // pairs (s, c) with value s - c in the order of the P_* slots
            float2 out[NPART];
#define KGS_SLOT(slot, pair, comp) out[slot] = make_float2(S[pair].s.comp, -S[pair].n.comp)
            KGS_SLOT(P_S0, 0, x);
            KGS_SLOT(P_S1X, 0, y);
            KGS_SLOT(P_S1Y, 1, x);
            KGS_SLOT(P_S1Z, 1, y);
            KGS_SLOT(P_S2YY, 2, x);
            KGS_SLOT(P_S2ZZ, 2, y);
            KGS_SLOT(P_S2XY, 3, x);
            KGS_SLOT(P_S2XZ, 3, y);
            KGS_SLOT(P_S2XX, 4, x);
            KGS_SLOT(P_S2YZ, 4, y);
            KGS_SLOT(P_S3Y, 5, x);
            KGS_SLOT(P_S3Z, 5, y);
            KGS_SLOT(P_S3X, 6, x);
            KGS_SLOT(P_FX, 6, y);
            KGS_SLOT(P_FY, 7, x);
            KGS_SLOT(P_FZ, 7, y);
#undef KGS_SLOT
            if (vp == 1) {
#pragma unroll
                for (int q = 0; q < NPART; q++) red[q * SLICE + cl] = out[q];
            }
            pair_barrier();
            if (vp == 0 && valid) {
                float2 *pp = COHERENT ? static_cast<float2 *>(scratch) + ((size_t)lk * SLICE + cl) * NPART
                                      : static_cast<float2 *>(a.part) +
                                            ((size_t)vgid * ncell + CELL(GX(li), GY(lj), z)) * NPART;
#pragma unroll
                for (int q = 0; q < NPART; q += 2) {
                    const float2 o0 = red[q * SLICE + cl], o1 = red[(q + 1) * SLICE + cl];
                    const float2 r0 = pair_add(out[q].x, out[q].y, o0.x, o0.y);
                    const float2 r1 = pair_add(out[q + 1].x, out[q + 1].y, o1.x, o1.y);
                    *reinterpret_cast<float4 *>(pp + q) = make_float4(r0.x, r0.y, r1.x, r1.y);
                }
            }
        }
        // the next slice's halo row overwrites the reduction buffer
        __syncthreads();
    }

    // z outflow of the block for the next stage (own velocities only)
    if (!zlast && ok) {
        for (int cl = 0; cl < SLICE; cl++) {
            const int li = cl % BX, lj = cl / BX;
            if (li >= ex || lj >= ey) continue;
            *reinterpret_cast<float2 *>(FZp + ((size_t)GY(lj) * nx + GX(li)) * Nv + gv) = slice[cl * CSP + t];
        }
    }
}

template <int LINE, bool UNIF>
__global__ void __launch_bounds__(NT, 2) sweep2_staged_kernel(const SweepArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    sweep_item2<LINE, false, UNIF, false>(a, a.work[blockIdx.x], blockIdx.y, smem, nullptr, nullptr);
}

template <int LINE, bool UNIF, bool DEV>
__global__ void __launch_bounds__(NT, 2) sweep2_persistent_kernel(const BatchSweepArgs b)
{
    extern __shared__ __align__(16) unsigned char smem[];
    persistent_loop<float>(b, [&](const SweepArgs &a, const int4 w, const int vg, void *scratch, Pipe &pipe) {
        sweep_item2<LINE, true, UNIF, DEV>(a, w, vg, smem, scratch, &pipe);
    });
}

using Persistent = void (*)(BatchSweepArgs);
Persistent pick(const SweepKind &k)
{
    if (k.dev) return k.line16 ? sweep2_persistent_kernel<16, true, true> : sweep2_persistent_kernel<0, true, true>;
    if (k.line16)
        return k.uniform ? sweep2_persistent_kernel<16, true, false> : sweep2_persistent_kernel<16, false, false>;
    return k.uniform ? sweep2_persistent_kernel<0, true, false> : sweep2_persistent_kernel<0, false, false>;
}

}  // namespace

size_t sweep2_smem_bytes(const SweepKind &k, int nxo_max) { return Layout2::total(nxo_max, k.line16 != 0, k.lines_max); }

int sweep2_occupancy(const SweepKind &k, size_t smem)
{
    int n = 0;
    const Persistent fn = pick(k);
    if (ensure_smem(reinterpret_cast<const void *>(fn), smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, NT, smem) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t launch_sweep2_persistent(const SweepKind &k, const BatchSweepArgs &b, int nxo_max, int grid,
                                     cudaStream_t s)
{
    const size_t smem = sweep2_smem_bytes(k, nxo_max);
    const Persistent fn = pick(k);
    const cudaError_t e = ensure_smem(reinterpret_cast<const void *>(fn), smem);
    if (e != cudaSuccess) return e;
    fn<<<grid, NT, smem, s>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_sweep2_staged(const SweepKind &k, const SweepArgs &a, int n_items, int max_vg, cudaStream_t s)
{
    void (*fn)(SweepArgs) = a.line16 ? (a.uniform ? sweep2_staged_kernel<16, true> : sweep2_staged_kernel<16, false>)
                                     : (a.uniform ? sweep2_staged_kernel<0, true> : sweep2_staged_kernel<0, false>);
    const size_t smem = sweep2_smem_bytes(k, a.nxo_max);
    const cudaError_t e = ensure_smem(reinterpret_cast<const void *>(fn), smem);
    if (e != cudaSuccess) return e;
    fn<<<dim3(n_items, max_vg), NT, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace kgs
