// kgs_conv_tc.cu -- 3x3x3 convolution as an implicit GEMM on the fifth-
// generation tensor cores (tcgen05.mma, accumulator in tensor memory).
//
// GEMM view: out[v][co] = sum over taps t and input channels ci of
// in[v + off(t)][ci] W[t][co][ci].  The unit of work is an 8 (x) by 16 (y)
// patch of two consecutive z-planes: two accumulators of M = 128 rows (voxels)
// each, all output channels (N = cout_p <= 112), so every weight tile that
// reaches shared memory feeds the MMAs of both planes.  One CTA per SM takes a
// contiguous range of units, z fastest, so that it marches up the columns of
// the volume: of a unit's four input planes (10 x 18 voxels, all channels
// each) the first two are the last two of the unit before.  The planes go
// through a ring of three slots in the K-major no-swizzle layout the MMA
// reads: 16-byte rows (8 channels of one voxel), x fastest within a channel
// octet, so that for every tap the 8 x positions of an output row segment are
// 8 consecutive 16-byte rows (one 8 x 16 B core matrix) and the 16 y rows and
// the channel octets are fixed strides.  Each tap is then C/16 MMAs of 128 x N
// x 16 per plane reading shifted windows of the staged planes; no im2col copy
// is made.  The weights, packed beforehand so that a tap is one contiguous
// block in the layout the MMA reads, move with one bulk copy per tap into a
// ring of four buffers.
//
// The warps have one role each, joined by barriers per slot and no CTA-wide
// ones: a producer issues the weight copies, an issuer the MMAs, five warps
// copy planes (cp.async, a slot ahead), and four warps read the accumulators
// of the previous unit with tcgen05.ld (two sets take turns in tensor memory)
// and apply bias + ReLU, bias only, or the ReLU mask of the backward pass.
// What bounds it: 112 -> 112 channels on 64^3 voxels take 125 us (1.42
// PFLOP/s), of which the MMAs are 76 us at their rate of 61 cycles; the rest
// is the weights' stream (12%) and the copies and epilogue beside it.  With a
// CTA per unit, which loaded its first planes before and read its
// accumulators after its MMAs, and one thread forming every descriptor anew,
// the layer took 222 us.
//
// The weight gradient (wgrad_tc_kernel) is the per-tap GEMM dW[t][co][ci] =
// sum over voxels v of dy[v][co] in[v + off(t)][ci], with the output
// channels in the 128 accumulator lanes (rows past Cout are ignored), the
// input channels as N and the voxels as the reduction dimension.  Both
// stored tensors keep the channels of a voxel contiguous, which for this GEMM
// is the MN-major operand layout (a core matrix is 8 voxels along K by 8
// channels in 16 bytes; instruction-descriptor bits 15 and 16), so tiles move
// with 16-byte cp.async and need no transpose.  A CTA takes the three taps
// that share (kz, ky): three accumulators in tensor memory, and per 8 x 16
// voxel tile one staged dy tile plus one 16 x 10 voxel block of input plane
// z + kz - 1 whose x windows at offsets 0, 1, 2 are the three B operands.
// A CTA covers a chunk of tiles of one sample and writes its partial; the
// caller sums the partials in a fixed order.
//
// Every wait on a barrier is bounded; on expiry the CTA records the error,
// waits (bounded) for its own MMAs, frees its tensor memory and returns.
#include <algorithm>
#include <cstdint>

#include "kgs_nn.h"

namespace kgs {
namespace nn {
namespace {

constexpr int TX = 8, TY = 16;                 // output patch: 128 voxels = 128 GEMM rows
constexpr int HX = TX + 2, HY = TY + 2, HZ = 3;  // input plane of the patch; ring of HZ plane slots
constexpr int OZ = 2;                          // output planes per step (two accumulators)
constexpr int TMEM_HALF = 128;                 // columns of one accumulator (>= N)
constexpr int TMEM_COLS = 2 * OZ * TMEM_HALF;  // two pairs in turn; a power of two
constexpr int FIRST_LOADER = 6;                // warps: producer, issuer, four of the epilogue, then the loaders
constexpr int LOADERS = 160;                   // threads that load input planes: a row of 10 x 14 pieces at least
constexpr int THREADS = FIRST_LOADER * 32 + LOADERS;
constexpr int NBUF = 4;                        // weight buffers: up to four taps in flight
constexpr long long WAIT_POLLS = 1ll << 20;    // try_wait polls before giving up

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: K-major operand without swizzling.
// lbo: bytes between core matrices adjacent along K; sbo: bytes between core
// matrices adjacent along M (or N).  Bits 46-47 hold the descriptor version
// (1 on this architecture family); base offset, LBO mode and layout type 0.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), bf16
// A and B (bits 7-9 and 10-12 = 1), both K-major (bits 15, 16 = 0), N / 8 in
// bits 17-22, M / 16 in bits 24-28.
__host__ __device__ constexpr uint32_t instr_desc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    for (long long i = 0; i < WAIT_POLLS; i++) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// 16-byte asynchronous global -> shared copy; zero-fills when !valid (no
// global read is made then; src must still be a valid address).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned)
// from global to shared memory; completion is counted on barrier `bar`.
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// MMA and commit are issued by one elected lane of a converged warp.  The
// whole warp runs the issuing loop so that descriptors and addresses stay in
// uniform registers, where the instruction takes them: from a branch of one
// thread they are moved there for every MMA, which then cost 128 cycles to
// issue against the 61 that the tensor core takes (128 x 112 x 16).
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
        : "memory");
}

__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

// Bounded wait of a whole warp.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity));
}

// The same for warps that also give up once another has (*fail, written while
// they run).  The flag goes into the vote: lanes that read different values
// must not part before a vote of all of them.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, const volatile int *fail)
{
    return __all_sync(0xffffffffu, *fail == 0 && mbar_wait(bar, parity));
}

// Warp index as a value that the compiler knows to be uniform.
__device__ __forceinline__ int uniform_warp() { return __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0); }

// Which 16-byte pieces of a voxel row a group of threads copies: eight threads
// take four channel octets of two neighbouring voxels, so that they read 64
// contiguous bytes per voxel and, with ten voxels per octet in shared memory,
// write to eight different 16-byte columns of the banks.
__host__ __device__ constexpr int row_threads(int X, int C8) { return X / 2 * ((C8 + 3) / 4) * 8; }
__device__ __forceinline__ void row_piece(int u, int X, int &x, int &c8)
{
    const int l = u % 8, g = u / 8;
    x = g % (X / 2) * 2 + l / 4;
    c8 = g / (X / 2) * 4 + l % 4;
}

// Weights W[t][co][ci] -> packed[t][ci/8][co][8]: each tap becomes one
// contiguous block in exactly the shared-memory layout the MMA reads, so it
// moves with a single bulk copy.
__global__ void pack_w_kernel(const uint4 *__restrict__ w, int cout_p, int c8n, uint4 *__restrict__ wpk)
{
    const size_t per = (size_t)cout_p * c8n;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 27 * per) return;
    const size_t t = i / per, r = i % per;
    const int co = (int)(r / c8n), c8 = (int)(r % c8n);
    wpk[t * per + (size_t)c8 * cout_p + co] = w[i];
}

// RES: the weights of all 27 taps fit beside the planes and are copied once
// per CTA; otherwise they stream through the ring, once per unit.
template <int MODE, bool RES>
__global__ void __launch_bounds__(THREADS, 1)
    conv_tc_kernel(const __nv_bfloat16 *__restrict__ in, const __nv_bfloat16 *__restrict__ wpk,
                   const float *__restrict__ bias, void *out, const __nv_bfloat16 *__restrict__ gate, ConvDims dm,
                   int *err)
{
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) uint64_t full_bar[NBUF], empty_bar[NBUF], plane_full[HZ], plane_empty[HZ], acc_full[2],
        acc_empty[2], done_bar;
    __shared__ uint32_t tmem_base;
    __shared__ int s_fail, s_last;  // a wait gave up; last weight copy whose MMAs were committed

    const int C8 = dm.cin_p / 8, cout_p = dm.cout_p;
    const uint32_t plane_bytes = (uint32_t)HY * C8 * HX * 16;
    const uint32_t w_bytes = (uint32_t)C8 * cout_p * 16;
    const int tiles_x = (dm.W + TX - 1) / TX, tiles = tiles_x * ((dm.H + TY - 1) / TY);
    const int pairs = (dm.D + OZ - 1) / OZ;  // plane pairs of a column (one patch of one sample)
    const long long units = (long long)dm.B * tiles * pairs;
    const long long u0 = units * blockIdx.x / gridDim.x, u1 = units * (blockIdx.x + 1) / gridDim.x;
    const int n_pairs = (int)(u1 - u0);
    const size_t vol = (size_t)dm.D * dm.H * dm.W;
    const int t = threadIdx.x, warp = uniform_warp(), lane = t % 32;
    const uint32_t halo_a = smem_u32(sm), w_a = halo_a + HZ * plane_bytes;
    volatile int *fail = &s_fail;  // written by the pipeline threads
    // weight copy T (pair T / 27 of this CTA, tap T % 27) goes through ring slot T % NBUF
    auto full = [&](int T) { return smem_u32(&full_bar[T % NBUF]); };    // weights landed
    auto empty = [&](int T) { return smem_u32(&empty_bar[T % NBUF]); };  // MMAs done
    auto use = [](int T) { return (uint32_t)((T / NBUF) & 1); };         // phase parity
    // plane n of this CTA's sequence goes through slot n % HZ
    auto pfull = [&](int n) { return smem_u32(&plane_full[n % HZ]); };
    auto pempty = [&](int n) { return smem_u32(&plane_empty[n % HZ]); };
    auto puse = [](int n) { return (uint32_t)((n / HZ) & 1); };
    // the pair starts a column: its four planes are new (else the last two of the pair before come first)
    auto fresh = [&](long long u) { return u == u0 || u % pairs == 0; };

    if (t == 0) {
        for (int q = 0; q < NBUF; q++) {
            mbar_init(smem_u32(&full_bar[q]), 1);
            mbar_init(smem_u32(&empty_bar[q]), 1);
        }
        for (int q = 0; q < HZ; q++) {
            mbar_init(smem_u32(&plane_full[q]), LOADERS);
            mbar_init(smem_u32(&plane_empty[q]), 1);
        }
        for (int q = 0; q < 2; q++) {
            mbar_init(smem_u32(&acc_full[q]), 1);
            mbar_init(smem_u32(&acc_empty[q]), 128);
        }
        mbar_init(smem_u32(&done_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = 0;
        s_last = -1;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base, 0);
    int issued = -1;  // last weight copy issued (thread 0)

    if (t == 0 && RES) {
        mbar_expect_tx(smem_u32(&full_bar[0]), 27 * w_bytes);
        for (int tap = 0; tap < 27; tap++)
            bulk_copy(w_a + (uint32_t)tap * w_bytes, wpk + (size_t)tap * cout_p * dm.cin_p, w_bytes,
                      smem_u32(&full_bar[0]));
        issued = 0;
    } else if (t == 0) {
        // weight producer: copy T reuses the slot of copy T - NBUF once its MMAs are done
        for (int T = 0; T < 27 * n_pairs; T++) {
            if (*fail || (T >= NBUF && !mbar_wait(empty(T - NBUF), use(T - NBUF)))) {
                *fail = 1;
                break;
            }
            mbar_expect_tx(full(T), w_bytes);
            bulk_copy(w_a + (uint32_t)(T % NBUF) * w_bytes, wpk + (size_t)(T % 27) * cout_p * dm.cin_p, w_bytes, full(T));
            issued = T;
        }
    } else if (warp == 1) {
        // MMA issuer: per tap and channel pair, one MMA of 128 x N x 16 for
        // each output plane, both reading the same weights.  Descriptors
        // advance by additions (their address field counts 16-byte units) and
        // ring slots by counters: with both formed anew for every MMA a step
        // of two MMAs took 300 cycles whatever its size.
        const uint32_t idesc = instr_desc(128, cout_p);
        const uint64_t a_desc = smem_desc(0, HX * 16, (uint32_t)C8 * HX * 16);
        const uint64_t b_desc = smem_desc(0, (uint32_t)cout_p * 16, 8 * 16), b_kc = 2 * (uint32_t)cout_p;
        const uint32_t halo16 = halo_a >> 4, plane16 = plane_bytes >> 4, row16 = (uint32_t)C8 * HX;
        const int KC = C8 / 2;
        int n0 = 0;                   // first plane of the pair: planes n0 .. n0 + 3
        int T = 0, slot = 0;          // weight copy (RES: tap), its ring slot
        uint32_t phase = 0;
        bool ok = true;
        if (RES) {
            ok = warp_wait(smem_u32(&full_bar[0]), 0);
            if (ok) T = 1;
        }
        for (int j = 0; j < n_pairs && ok; j++) {
            if (j > 0) n0 += fresh(u0 + j) ? 4 : 2;
            const bool end = j + 1 == n_pairs || fresh(u0 + j + 1);  // the column ends here
            const uint32_t acc = tmem + (uint32_t)((j & 1) * OZ * TMEM_HALF);
            // the accumulators of pair j - 2 have been read
            if (j >= 2) ok = warp_wait(smem_u32(&acc_empty[j & 1]), (uint32_t)((j - 2) / 2 & 1));
            ok = ok && warp_wait(pfull(n0), puse(n0));
            uint32_t first = 0;  // the pair's first MMA overwrites its accumulator
            for (int kz = 0; kz < 3 && ok; kz++) {
                ok = warp_wait(pfull(n0 + kz + 1), puse(n0 + kz + 1));
                tc_fence_after();
                const uint64_t pa0 = a_desc + halo16 + (uint32_t)((n0 + kz) % HZ) * plane16;      // output z0
                const uint64_t pa1 = a_desc + halo16 + (uint32_t)((n0 + kz + 1) % HZ) * plane16;  // output z0 + 1
                for (int ky = 0; ky < 3 && ok; ky++)
                    for (int kx = 0; kx < 3; kx++) {
                        if (!RES) {
                            if (!ok || !warp_wait(smem_u32(&full_bar[slot]), phase)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                        }
                        uint64_t d0 = pa0 + (uint32_t)ky * row16 + kx, d1 = pa1 + (uint32_t)ky * row16 + kx;
                        uint64_t bd = b_desc + ((w_a + (uint32_t)(RES ? 9 * kz + 3 * ky + kx : slot) * w_bytes) >> 4);
                        for (int kc = 0; kc < KC; kc++) {
                            tc_mma(acc, d0, bd, idesc, first | (uint32_t)kc);
                            tc_mma(acc + TMEM_HALF, d1, bd, idesc, first | (uint32_t)kc);
                            d0 += 2 * HX;
                            d1 += 2 * HX;
                            bd += b_kc;
                        }
                        first = 1;
                        if (!RES) {
                            tc_commit(smem_u32(&empty_bar[slot]));
                            T++;
                            if (++slot == NBUF) slot = 0, phase ^= 1;
                        }
                    }
                if (!ok) break;
                // planes that no later MMA reads
                if (kz < 2) {
                    tc_commit(pempty(n0 + kz));
                } else if (end) {
                    tc_commit(pempty(n0 + 2));
                    tc_commit(pempty(n0 + 3));
                }
            }
            if (ok) tc_commit(smem_u32(&acc_full[j & 1]));
        }
        // all MMAs of the CTA are complete once the done barrier has fired
        tc_commit(smem_u32(&done_bar));
        ok = warp_wait(smem_u32(&done_bar), 0) && ok;
        if (lane == 0) {
            s_last = T - 1;
            if (!ok) *fail = 1;
        }
    } else if (warp >= FIRST_LOADER) {
        // loaders: a thread keeps its (x, channel octet) and walks down the
        // rows of a plane; whole rows per pass
        const int lt = t - FIRST_LOADER * 32, per = row_threads(HX, C8), rows = LOADERS / per;
        int px, c8;
        row_piece(lt % per, HX, px, c8);
        const int r0 = lt / per;
        const bool idle = r0 >= rows || c8 >= C8;
        int n = 0;
        bool ok = true;
        auto load = [&](long long u, int p) {  // plane z0 - 1 + p of unit u as plane n
            const long long col = u / pairs;
            const int patch = (int)(col % tiles), b = (int)(col / tiles);
            const int z = (int)(u % pairs) * OZ - 1 + p;
            const int x = patch % tiles_x * TX - 1 + px, y = patch / tiles_x * TY - 1 + r0;
            if (idle) return;
            const bool plane = x >= 0 && x < dm.W && z >= 0 && z < dm.D;
            const __nv_bfloat16 *src =
                in + ((long long)b * (long long)vol + ((long long)z * dm.H + y) * dm.W + x) * dm.cin_p + c8 * 8;
            uint32_t dst = halo_a + (uint32_t)(n % HZ) * plane_bytes + (uint32_t)((r0 * C8 + c8) * HX + px) * 16;
            for (int r = r0, yy = y; r < HY; r += rows, yy += rows) {
                const bool in_y = plane && yy >= 0 && yy < dm.H;
                cp_async16(dst, in_y ? src : in, in_y);
                src += (long long)rows * dm.W * dm.cin_p;
                dst += (uint32_t)(rows * C8 * HX) * 16;
            }
        };
        for (long long u = u0; u < u1 && ok; u++) {
            for (int p = fresh(u) ? 0 : 2; p < 4; p++, n++) {
                // plane n reuses the slot of plane n - HZ once no MMA reads it
                if (n >= HZ && !warp_wait(pempty(n - HZ), puse(n - HZ), fail)) {
                    *fail = 1;  // the issuer's wait on this plane then gives up too
                    ok = false;
                    break;
                }
                load(u, p);
                cp_async_commit();
                // the first HZ planes are issued together, the later ones one per nine taps
                if (n < HZ - 1) continue;
                if (n == HZ - 1) {
                    static_assert(HZ == 3, "two planes are outstanding before this one");
                    cp_async_wait<2>();
                    fence_async_smem();
                    mbar_arrive(pfull(0));
                    cp_async_wait<1>();
                    fence_async_smem();
                    mbar_arrive(pfull(1));
                }
                cp_async_wait<0>();
                fence_async_smem();
                mbar_arrive(pfull(n));
            }
        }
        cp_async_wait<0>();
    } else if (warp >= 2) {
        // epilogue warps 2 .. 5: warp w reads the TMEM lanes 32 (w % 4) ..
        // (output rows) while the MMAs of the next pair run
        const int quad = warp % 4, row = quad * 32 + lane;
        for (int j = 0; j < n_pairs; j++) {
            if (!warp_wait(smem_u32(&acc_full[j & 1]), (uint32_t)(j / 2 & 1), fail)) {
                *fail = 1;
                break;
            }
            tc_fence_after();
            const long long u = u0 + j, col = u / pairs;
            const int patch = (int)(col % tiles), b = (int)(col / tiles), z0 = (int)(u % pairs) * OZ;
            const int vx = patch % tiles_x * TX + row % TX, vy = patch / tiles_x * TY + row / TX;
            const bool inside = vx < dm.W && vy < dm.H;
            const uint32_t acc = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)((j & 1) * OZ * TMEM_HALF);
            for (int oz = 0; oz < OZ; oz++) {
                const int z = z0 + oz;
                if (z >= dm.D) break;  // uniform over the CTA
                const size_t vo = (size_t)b * vol + ((size_t)z * dm.H + vy) * dm.W + vx;
                for (int c0 = 0; c0 < cout_p; c0 += 16) {
                    float v[16];
                    __syncwarp();  // lanes outside the volume skip the stores
                    tc_ld16(acc + (uint32_t)(oz * TMEM_HALF + c0), v);  // all lanes
                    if (!inside) continue;
                    if (MODE == 1) {
                        float *o = static_cast<float *>(out) + vo * cout_p + c0;
#pragma unroll
                        for (int i = 0; i < 16; i += 4)
                            *reinterpret_cast<float4 *>(o + i) =
                                make_float4(v[i] + bias[c0 + i], v[i + 1] + bias[c0 + i + 1],
                                            v[i + 2] + bias[c0 + i + 2], v[i + 3] + bias[c0 + i + 3]);
                    } else {
                        __align__(16) __nv_bfloat162 h[8];
                        if (MODE == 0) {
#pragma unroll
                            for (int i = 0; i < 8; i++)
                                h[i] = __floats2bfloat162_rn(fmaxf(v[2 * i] + bias[c0 + 2 * i], 0.f),
                                                             fmaxf(v[2 * i + 1] + bias[c0 + 2 * i + 1], 0.f));
                        } else {
                            __align__(16) __nv_bfloat162 g[8];
                            const uint4 *gp = reinterpret_cast<const uint4 *>(gate + vo * cout_p + c0);
                            reinterpret_cast<uint4 *>(g)[0] = gp[0];
                            reinterpret_cast<uint4 *>(g)[1] = gp[1];
#pragma unroll
                            for (int i = 0; i < 8; i++)
                                h[i] = __floats2bfloat162_rn(__bfloat162float(g[i].x) > 0.f ? v[2 * i] : 0.f,
                                                             __bfloat162float(g[i].y) > 0.f ? v[2 * i + 1] : 0.f);
                        }
                        uint4 *o = reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(out) + vo * cout_p + c0);
                        o[0] = reinterpret_cast<uint4 *>(h)[0];
                        o[1] = reinterpret_cast<uint4 *>(h)[1];
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(smem_u32(&acc_empty[j & 1]));
        }
    }
    __syncthreads();  // the pipeline has ended; the outcome in s_fail is uniform after it
    if (t == 0 && s_fail) {
        atomicExch(err, 1);
        // weight copies issued but never consumed land before the CTA
        // leaves (bounded; at most NBUF are outstanding, on distinct barriers)
        for (int T = s_last + 1; T <= issued; T++) (void)mbar_wait(full(T), use(T));
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// ---------------------------------------------------------------------------
// Weight gradient: part[b][chunk][t][co][ci] = sum over the chunk's voxels v
// of dy[v][co] * in[v + off(t)][ci], per tap a tcgen05 GEMM with M = co (128
// TMEM lanes, rows >= cout_p ignored), N = ci and K = voxels in steps of 16.
// Both tensors store the channels of a voxel contiguously, which for this
// GEMM is the MN-major operand layout: a core matrix is 8 voxels (along K) x
// 8 channels (16 bytes), so tiles move with 16-byte asynchronous copies and
// need no transpose.  A CTA takes the three taps that share (kz, ky) -- three
// accumulators in tensor memory -- for a chunk of 8 x 16-voxel tiles.  Per
// tile it stages dy of the tile, [y][co/8][x of 10][16 B], and rows y0 + ky - 1 ..
// y0 + ky + 14, columns x0 - 1 .. x0 + 8 of input plane z + kz - 1,
// [y][ci/8][x][16 B]; the windows of that block at x offsets 0, 1, 2 are the
// B operands of the three taps.
//
// What bounds it: the copies.  A tile brings 64 KB for 24 MMAs of 128 x 112 x
// 16 (1500 cycles of the tensor core), because tensor memory holds three taps'
// accumulators and the nine (kz, ky) read the tiles again: 0.8 GB through L2
// for a 112 -> 112 layer on 4 x 32^3 voxels in 117 us, 52% of the L2's rate
// with the tensor core 40% busy (288 CTAs are 1.9 waves of 152 SMs); 305 us on
// 8 x 32^3.  Nine warps
// only copy and one only issues MMAs, through barriers per tile buffer, so
// neither waits for the other beyond the three buffers; a copying thread
// keeps its (x, channel octet) from tile to tile and walks down the rows by
// adding one stride.  With CTA barriers between copies and MMAs and the place
// of every 16-byte piece recomputed by divisions the layer took 490 us, and a
// 16 -> 48 one 297 us instead of 107.
constexpr int WG_BUF = 3;           // tile buffers
constexpr int WG_TMEM = 512;        // three accumulators of 128 columns
constexpr int WG_COPY = 288;        // copying threads: warps 0 .. 8
constexpr int WG_THREADS = WG_COPY + 32;  // and the warp of the MMA thread

// Voxel tiles of 128 per CTA: chunks as long as 32 tiles, shorter ones where
// the device would otherwise have fewer than one CTA per SM (8 x 16^3: 72
// CTAs of 32 tiles against 144 of 16).
int wg_tiles_per_cta(const ConvDims &dm)
{
    const int tiles = ((dm.W + TX - 1) / TX) * ((dm.H + TY - 1) / TY) * dm.D;
    int n = 32;
    while (n > 4 && 9ll * dm.B * ((tiles + n - 1) / n) < 140) n /= 2;
    return n;
}

// kind::f16 instruction descriptor with both operands MN-major (bits 15, 16).
__host__ __device__ constexpr uint32_t instr_desc_mn(int M, int N)
{
    return instr_desc(M, N) | (1u << 15) | (1u << 16);
}

struct WgLayout {
    uint32_t a_bytes, h_bytes, buf_bytes, total;
};
// Shared memory of the weight-gradient CTA: WG_BUF x (dy tile, input block).
// The MMA reads 16 octets of dy where there are cout_p / 8; the excess lies in
// the input block behind it and feeds accumulator rows that are not stored.
__host__ __device__ inline WgLayout wg_layout(int cin_p, int cout_p)
{
    const int c8o = cout_p / 8, c8i = cin_p / 8;
    WgLayout L;
    L.a_bytes = (uint32_t)(TY * c8o * HX * 16);  // eight voxels in the room of HX (row_piece)
    L.h_bytes = (uint32_t)(TY * c8i * HX * 16);
    L.buf_bytes = L.a_bytes + L.h_bytes;
    L.total = WG_BUF * L.buf_bytes + 128;
    return L;
}

__global__ void __launch_bounds__(WG_THREADS, 1)
    wgrad_tc_kernel(const __nv_bfloat16 *__restrict__ in, const __nv_bfloat16 *__restrict__ dy,
                    float *__restrict__ part, ConvDims dm, int n_chunks, int tiles_per_cta, int *err)
{
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) uint64_t full_bar[WG_BUF], empty_bar[WG_BUF], done_bar;
    __shared__ uint32_t tmem_base;
    __shared__ int s_fail;
    const int cout_p = dm.cout_p, cin_p = dm.cin_p, C8o = cout_p / 8, C8i = cin_p / 8;
    const WgLayout L = wg_layout(cin_p, cout_p);
    const uint32_t base = smem_u32(sm);
    const int g = blockIdx.x, chunk = blockIdx.y, b = blockIdx.z;
    const int kz = g / 3, ky = g % 3;  // taps 9 kz + 3 ky + kx, kx = 0, 1, 2
    const int tiles_x = (dm.W + TX - 1) / TX, tiles_y = (dm.H + TY - 1) / TY;
    const int n_tiles = tiles_x * tiles_y * dm.D;
    const int tile0 = chunk * tiles_per_cta, nt = min(n_tiles, tile0 + tiles_per_cta) - tile0;
    const size_t vol = (size_t)dm.D * dm.H * dm.W;
    const int t = threadIdx.x, warp = uniform_warp(), lane = t % 32;
    volatile int *fail = &s_fail;

    if (t == 0) {
        for (int q = 0; q < WG_BUF; q++) {
            mbar_init(smem_u32(&full_bar[q]), WG_COPY);
            mbar_init(smem_u32(&empty_bar[q]), 1);
        }
        mbar_init(smem_u32(&done_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(WG_TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base, 0);

    if (warp < WG_COPY / 32) {
        // The copying threads split in two parts, one per tensor, in the ratio
        // of their pieces; a part covers whole voxel rows of its block at a
        // time, a thread one (x, octet) of them.
        const int na = row_threads(TX, C8o), nh = row_threads(HX, C8i);
        const int ra = WG_COPY / (na + nh);             // rows of the dy tile per pass (na + nh <= 288)
        const int rh = (WG_COPY - ra * na) / nh;        // rows of the input block per pass
        const bool is_a = t < ra * na;
        const int u = is_a ? t : t - ra * na;
        const int per = is_a ? na : nh, rows = is_a ? ra : rh, C8 = is_a ? C8o : C8i;
        int px, c8;
        row_piece(u % per, is_a ? TX : HX, px, c8);
        const int r0 = u / per;
        const bool idle = r0 >= rows || c8 >= C8;
        const uint32_t s_off = (is_a ? 0u : L.a_bytes) + (uint32_t)((r0 * C8 + c8) * HX + px) * 16;
        const uint32_t s_step = (uint32_t)(rows * C8 * HX) * 16;
        const int cp = is_a ? cout_p : cin_p;
        const __nv_bfloat16 *tensor = (is_a ? dy : in) + (size_t)b * vol * cp + c8 * 8;
        const long long g_step = (long long)rows * dm.W * cp;
        for (int i = 0; i < nt; i++) {
            // tile i reuses the buffer of tile i - WG_BUF: its MMAs must have completed
            if (i >= WG_BUF && !warp_wait(smem_u32(&empty_bar[i % WG_BUF]), (uint32_t)(i / WG_BUF - 1) & 1, fail)) {
                *fail = 1;
                break;
            }
            const int tile = tile0 + i;
            const int tz = tile / (tiles_x * tiles_y), txy = tile % (tiles_x * tiles_y);
            const int x = (txy % tiles_x) * TX + px - (is_a ? 0 : 1);
            const int y = (txy / tiles_x) * TY + r0 + (is_a ? 0 : ky - 1), z = tz + (is_a ? 0 : kz - 1);
            if (!idle) {
                const bool plane = x >= 0 && x < dm.W && z >= 0 && z < dm.D;
                const __nv_bfloat16 *src = tensor + (((long long)z * dm.H + y) * dm.W + x) * cp;
                uint32_t dst = base + (uint32_t)(i % WG_BUF) * L.buf_bytes + s_off;
                for (int r = r0, yy = y; r < TY; r += rows, yy += rows, src += g_step, dst += s_step) {
                    const bool ok = plane && yy >= 0 && yy < dm.H;
                    cp_async16(dst, ok ? src : tensor, ok);
                }
            }
            cp_async_commit();
            if (i >= 1) {  // tile i - 1 has landed, while tile i is on its way
                cp_async_wait<1>();
                fence_async_smem();
                mbar_arrive(smem_u32(&full_bar[(i - 1) % WG_BUF]));
            }
        }
        cp_async_wait<0>();
        fence_async_smem();
        if (nt > 0 && !*fail) mbar_arrive(smem_u32(&full_bar[(nt - 1) % WG_BUF]));
    } else {
        // descriptors advance by additions (16-byte units), as in conv_tc_kernel
        const uint32_t idesc = instr_desc_mn(128, cin_p);
        const uint64_t a_desc = smem_desc(0, (uint32_t)(C8o * HX * 16), HX * 16), a_ks = 2 * C8o * HX;
        const uint64_t b_desc = smem_desc(0, (uint32_t)(C8i * HX * 16), HX * 16), b_ks = 2 * C8i * HX;
        uint32_t first = 0;
        bool ok = true;
        int slot = 0;
        uint32_t phase = 0;
        for (int i = 0; i < nt; i++) {
            ok = warp_wait(smem_u32(&full_bar[slot]), phase);
            if (!ok) break;
            tc_fence_after();
            const uint32_t abuf = base + (uint32_t)slot * L.buf_bytes;
            uint64_t ad = a_desc + (abuf >> 4), bd = b_desc + ((abuf + L.a_bytes) >> 4);
            for (int ks = 0; ks < TY / 2; ks++) {  // K = 16 voxels: tile rows 2ks, 2ks + 1
                tc_mma(tmem, ad, bd, idesc, first);
                tc_mma(tmem + 128, ad, bd + 1, idesc, first);
                tc_mma(tmem + 256, ad, bd + 2, idesc, first);
                first = 1;
                ad += a_ks;
                bd += b_ks;
            }
            tc_commit(smem_u32(&empty_bar[slot]));
            if (++slot == WG_BUF) slot = 0, phase ^= 1;
        }
        // every MMA issued has completed once the done barrier fires
        tc_commit(smem_u32(&done_bar));
        ok = warp_wait(smem_u32(&done_bar), 0) && ok;
        if (lane == 0 && !ok) *fail = 1;
    }
    __syncthreads();  // the other threads wait here, not polling; s_fail is uniform after it
    tc_fence_after();
    if (s_fail) {
        if (t == 0) atomicExch(err, 1);
    } else if (warp < 8) {
        // row co = TMEM lane (warps w and w + 4 share the lanes 32 (w % 4) ..
        // and take every other block of 16 columns); columns kx * 128 + ci
        const int co = (warp % 4) * 32 + lane, nb = cin_p / 16;
        for (int q = warp / 4; q < 3 * nb; q += 2) {
            const int kx = q / nb, c0 = q % nb * 16;
            float v[16];
            __syncwarp();  // lanes without a channel skip the stores
            tc_ld16(tmem + ((uint32_t)((warp % 4) * 32) << 16) + (uint32_t)(kx * 128 + c0), v);
            if (co >= cout_p) continue;
            float *dst = part + ((((size_t)b * n_chunks + chunk) * 27 + (kz * 3 + ky) * 3 + kx) * cout_p + co) * cin_p + c0;
#pragma unroll
            for (int k = 0; k < 16; k += 4)
                *reinterpret_cast<float4 *>(dst + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(WG_TMEM) : "memory");
    }
}

template <int MODE, bool RES>
cudaError_t launch(size_t smem, const __nv_bfloat16 *in, const __nv_bfloat16 *wpk, const float *bias, void *out,
                   const __nv_bfloat16 *gate, ConvDims dm, int *err, cudaStream_t s)
{
    // at least 120 KB: one CTA per SM, so no CTA waits for tensor memory held by another
    smem = std::max<size_t>(smem, 120 * 1024);
    int dev = 0, sms = 0;
    cudaError_t e =
        cudaFuncSetAttribute(conv_tc_kernel<MODE, RES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess || (e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    const long long units =
        (long long)((dm.W + TX - 1) / TX) * ((dm.H + TY - 1) / TY) * ((dm.D + OZ - 1) / OZ) * dm.B;
    conv_tc_kernel<MODE, RES><<<(unsigned)std::min<long long>(sms, units), THREADS, smem, s>>>(in, wpk, bias, out, gate,
                                                                                            dm, err);
    return cudaGetLastError();
}

// All taps' weights stay in shared memory where they fit (16 -> 48 and 48 -> 16
// channels): streamed again for every unit, their small copies are bound by
// latency (64^3 voxels: 16 -> 48 channels 73 us, 48 -> 16 97 us streamed).
template <int MODE>
cudaError_t launch(const __nv_bfloat16 *in, const __nv_bfloat16 *wpk, const float *bias, void *out,
                   const __nv_bfloat16 *gate, ConvDims dm, int *err, cudaStream_t s)
{
    const size_t planes = (size_t)HZ * HY * (dm.cin_p / 8) * HX * 16, tap = (size_t)(dm.cin_p / 8) * dm.cout_p * 16;
    if (planes + 27 * tap <= 220 * 1024)
        return launch<MODE, true>(planes + 27 * tap, in, wpk, bias, out, gate, dm, err, s);
    return launch<MODE, false>(planes + NBUF * tap, in, wpk, bias, out, gate, dm, err, s);
}

}  // namespace

cudaError_t conv_tc(int mode, const __nv_bfloat16 *in, const __nv_bfloat16 *w, __nv_bfloat16 *wpk, const float *bias,
                    void *out, const __nv_bfloat16 *gate, ConvDims dm, int *err, cudaStream_t s)
{
    if (dm.cin_p % 16 || dm.cout_p % 16 || dm.cin_p < 16 || dm.cout_p < 16 || dm.cin_p > 112 || dm.cout_p > 112)
        return cudaErrorInvalidValue;
    const size_t n16 = (size_t)27 * dm.cout_p * (dm.cin_p / 8);
    pack_w_kernel<<<(unsigned)((n16 + 255) / 256), 256, 0, s>>>(reinterpret_cast<const uint4 *>(w), dm.cout_p,
                                                                 dm.cin_p / 8, reinterpret_cast<uint4 *>(wpk));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    switch (mode) {
    case 0: return launch<0>(in, wpk, bias, out, gate, dm, err, s);
    case 1: return launch<1>(in, wpk, bias, out, gate, dm, err, s);
    default: return launch<2>(in, wpk, bias, out, gate, dm, err, s);
    }
}

int wgrad_chunks(const ConvDims &dm)
{
    const int tiles = ((dm.W + TX - 1) / TX) * ((dm.H + TY - 1) / TY) * dm.D;
    const int per = wg_tiles_per_cta(dm);
    return (tiles + per - 1) / per;
}

cudaError_t wgrad_tc(const __nv_bfloat16 *in, const __nv_bfloat16 *dy, float *part, ConvDims dm, int *err,
                     cudaStream_t s)
{
    if (dm.cin_p % 16 || dm.cout_p % 16 || dm.cin_p < 16 || dm.cout_p < 16 || dm.cin_p > 112 || dm.cout_p > 112)
        return cudaErrorInvalidValue;
    // at least 120 KB: one CTA per SM, so no CTA waits for tensor memory held by another
    const size_t smem = std::max<size_t>(wg_layout(dm.cin_p, dm.cout_p).total, 120 * 1024);
    cudaError_t e = cudaFuncSetAttribute(wgrad_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int n_chunks = wgrad_chunks(dm);
    wgrad_tc_kernel<<<dim3(9, n_chunks, dm.B), WG_THREADS, smem, s>>>(in, dy, part, dm, n_chunks,
                                                                      wg_tiles_per_cta(dm), err);
    return cudaGetLastError();
}

}  // namespace nn
}  // namespace kgs
