// kgs_sweep_d.cu -- the first-order FP64 sweep with separated equilibria
// (arXiv 1810.00348, Eqs. (2), (5), (7), (9)).  The work decomposition is that
// of kgs_sweep.cu; what differs is how an item is worked through.
//
// What bounds it.  One FP64 instruction of a warp occupies the scheduler's
// FP64 pipe for 64 cycles, dependent or not (two lanes per clock and SM), so a
// single warp per scheduler keeps the pipe busy and the time is the number of
// FP64 instructions per phase point; loads, addresses and integer work run in
// their shadow.  The kernel therefore trades FP64 operations for table
// entries, from 44 per phase point to about 18:
//
//  * On the tensor-product velocity grid the Maxwellian is a product of one
//    factor per axis, and the Shakhov factor is 1 + a b with a and b sums of
//    one term per axis.  With x against (y, z) as the split,
//      f^S/tau = E_x E_l (1 + (a_x + a_l)(b_x + b_l)) = sum_{r<4} G_r(x) H_r(l),
//      G = E_x {1 + a_x b_x, a_x, b_x, 1},  H = E_l {1, b_l, a_l, a_l b_l}:
//    four operations instead of an exponential and two inner products (28).
//    axis_kernel tabulates G per (cell, x node) and the y and z factors per
//    (cell, node) once per iteration (0.4% of the sweep's operations at 32
//    nodes per axis); a block forms H for the lines of its group, slice by
//    slice, in shared memory.
//  * f = num / den from the hardware reciprocal r (relative error below
//    2^-20): with e = 1 - den r, f = q + q (e + e^2), q = num r, is off by
//    e^3: four operations instead of six.
//  * The moment sums of a slice are about one velocity C, the middle of the
//    range of U^n over its fluid cells, so that the weights of a node are table
//    entries: four multiply-adds per velocity for P_a = sum w_x (xi_x - C_x)^a f
//    along a line, 16 per line for the 13 sums.  The sums kernel shifts them to
//    U^n, which costs no digits while U^n is near C.  A slice over which U^n
//    varies by more than CENTRE_RANGE of the thermal speed either way (a shock,
//    the front of a body) is summed about each cell's own U^n: eight operations
//    per velocity, 24 per line.  About 0 the shift subtracts terms of size
//    rho |U|^3, which left the heat flux of a Mach 2 stream 17 times and of a
//    Mach 5 stream 280 times further off.  The incoming wall flux of an octant
//    along d is its first moment along d up to sign.
//
// Cells are visited row by row: with the pipe saturated by one chain there is
// nothing to gain from independent cells.
//
// Measured: 32^3 cells x 32^3 velocities 87.2 -> 35.7 ms (30.7 ms are the 18
// operations at the pipe's rate), 27x19x22 x 17x14x20 19.3 -> 4.0 ms (with the
// overlap of neighbouring blocks).  Error of the heat flux against extended
// precision as with every sum about U^n: 8.4e-16 (8.6e-16) around a cube at
// Mach 2, 4.1e-14 (4.2e-14) in a Mach 2 stream, 1.3e-13 (1.6e-13) at Mach 5.
#include "kgs_sweep_dev.cuh"

namespace kgs {
namespace {

constexpr int VG = NT;           // velocities per group
constexpr int CS = VG + 1;       // odd stride of a cell: conflict-free per-cell reads
constexpr int HCOL = SLICE, HROW = SLICE + BY, NPOS = SLICE + BY + BX;
// Weights of a line: W = w_y w_z, Wy, Wz, Wyy, Wzz, Wyz, Wr, Wry, Wrz (r = y^2 + z^2;
// y and z about the slice's centre), xi_y.  These tables are as small as they
// can be: with 10 nodes per line (20 along x) two blocks fit an SM with 64
// bytes to spare, and one block alone takes 1.4 times as long.
constexpr int LW = 10;
// Largest distance of U^n from the centre of its slice, in thermal speeds of
// the coldest cell: at 1/8 the sums are as exact as about U^n itself (heat
// flux off by 1.0 to 1.1 times as much over random fields), at 0.45 1.8 times.
constexpr float CENTRE_RANGE = 0.125f;
static_assert(BX * CS >= NPART * SLICE, "reduction buffer in the halo row");

struct LayoutD {
    static constexpr size_t off_cell = align16(sizeof(double) * NPOS * CS);  // [SLICE][4] 1/tau, 1/dx, 1/dy, 1/dz
    static constexpr size_t off_flag = off_cell + sizeof(double) * SLICE * 4;
    static constexpr size_t off_cen = off_flag + sizeof(int) * SLICE;         // [2][4] centre of this and the next slice
    static constexpr size_t off_x = off_cen + sizeof(double) * 8;             // [nxm][4] w_x (xi_x - C_x)^a
    __host__ __device__ static size_t off_xi(int nxm) { return off_x + sizeof(double) * 4 * nxm; }  // [nxm] xi_x
    __host__ __device__ static size_t off_line(int nxm) { return off_xi(nxm) + align16(sizeof(double) * nxm); }
    __host__ __device__ static size_t off_h(int nxm, int lines_max)           // [SLICE][lines_max][4]
    {
        return off_line(nxm) + align16(sizeof(double) * LW * lines_max);
    }
    static size_t total(int nxm, int lines_max)
    {
        return off_h(nxm, lines_max) + sizeof(double) * 4 * SLICE * lines_max;
    }
};

// One record per (cell, node): x nodes G, y nodes {E_y, a_y, b_y, -}, z nodes
// {kappa E_z, a_z, b_z, -}, where f^S/tau = kappa E_x E_y E_z (1 + a b) and
// E = exp(-(xi^2 - 2 U xi) / (2RT)), a = c.q', b = |c|^2/(RT) - 5 as in
// coef_kernel, whose record it reads.
__global__ void __launch_bounds__(256)
    axis_kernel(const double *__restrict__ coef, const double *__restrict__ nodes, size_t ncell, int nvx, int nvy,
                int na, double4 *__restrict__ tab)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ncell * na) return;
    const size_t c = i / na;
    const int k = (int)(i % na);
    const double *r = coef + c * NCOEF;
    const int d = k < nvx ? 0 : k < nvx + nvy ? 1 : 2;
    const double x = nodes[k];
    const double s = x * (x + r[C_M2UX + d]);
    const double E = exp(s * r[C_NEXP]);
    double a = x * r[C_QX + d], b = s * r[C_RT1];
    double4 out;
    if (d == 0) {
        a += r[C_MUQ];
        b += r[C_SHK0];
        out = make_double4(fma(E * a, b, E), E * a, E * b, E);
    } else {
        out = make_double4(d == 2 ? E * r[C_KAPPA] : E, a, b, 0.0);
    }
    tab[i] = out;
}

// SweepArgs::centre: the middle of the range of U^n over the fluid cells of
// each block's slice (0 without any), and whether U^n is too far from it
// (CENTRE_RANGE) somewhere.  In FP32: any velocity near U^n will do, and the
// FP64 pipe takes 3 us for the comparisons.
__global__ void __launch_bounds__(SLICE)
    centre_kernel(const double *__restrict__ coef, int nx, int ny, double *__restrict__ centre)
{
    __shared__ float lo[4][2], hi[4][2];
    const int nbx = (nx + BX - 1) / BX, nby = (ny + BY - 1) / BY;
    const int bx = blockIdx.x % nbx, by = blockIdx.x / nbx % nby, k = blockIdx.x / (nbx * nby);
    const int t = threadIdx.x, i = bx * BX + t % BX, j = by * BY + t / BX;
    const double *r = coef + ((size_t)i + (size_t)nx * (j + (size_t)ny * k)) * NCOEF;
    const bool fluid = i < nx && j < ny && !(flag_bits(r[C_FLAGS]) & F_SOLID);
    for (int d = 0; d < 4; d++) {  // U^n along the axes, 1/(RT)
        const float v = fluid ? (d < 3 ? -0.5f * (float)r[C_M2UX + d] : (float)r[C_RT1]) : 0.f;
        float a = fluid ? v : INFINITY, b = fluid ? v : -INFINITY;
        for (int off = 16; off > 0; off >>= 1) {
            a = fminf(a, __shfl_xor_sync(0xffffffffu, a, off));
            b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, off));
        }
        if (t % 32 == 0) lo[d][t / 32] = a, hi[d][t / 32] = b;
    }
    __syncthreads();
    if (t > 0) return;
    float far2 = 0.f;
    double *out = centre + (size_t)blockIdx.x * 4;
    for (int d = 0; d < 3; d++) {
        const float a = fminf(lo[d][0], lo[d][1]), h = 0.5f * (fmaxf(hi[d][0], hi[d][1]) - a);
        out[d] = h >= 0.f ? a + h : 0.f;
        far2 += h * h;
    }
    const float rt1 = fmaxf(hi[3][0], hi[3][1]);  // of the coldest cell, thermal speed^2 = 2 / rt1
    out[3] = rt1 > 0.f && !(far2 * rt1 <= 2.f * CENTRE_RANGE * CENTRE_RANGE) ? 1.0 : 0.0;
}

__device__ __forceinline__ double4 ld_rec(const double4 *p)
{
    const double2 *q = reinterpret_cast<const double2 *>(p);
    const double2 u = __ldg(q), v = __ldg(q + 1);
    return make_double4(u.x, u.y, v.x, v.y);
}

template <bool UNIF>
__device__ __forceinline__ void sweep_item_d(const SweepArgs &a, const int4 w, const int vgy, unsigned char *smem,
                                             double *scratch, Pipe &pipe, const int lines_max)
{
    double *slice = reinterpret_cast<double *>(smem);
    double *cell4 = reinterpret_cast<double *>(smem + LayoutD::off_cell);
    int *cflag = reinterpret_cast<int *>(smem + LayoutD::off_flag);
    double *cen2 = reinterpret_cast<double *>(smem + LayoutD::off_cen);
    double *wxp = reinterpret_cast<double *>(smem + LayoutD::off_x);
    double *xi_x = reinterpret_cast<double *>(smem + LayoutD::off_xi(a.nxo_max));
    double *lw = reinterpret_cast<double *>(smem + LayoutD::off_line(a.nxo_max));
    double *H = reinterpret_cast<double *>(smem + LayoutD::off_h(a.nxo_max, lines_max));
    double *red = slice + HROW * CS;  // [NPART][SLICE]: the halo row is not read during the moment phase

    const int t = threadIdx.x;
    const int o = w.x;
    const int vcount = a.oct_vcount[o];
    const int v0 = vgy * VG;
    if (v0 >= vcount) return;
    const int nvg = min(VG, vcount - v0);
    const int nxo = a.oct_nx[o], nyo = a.oct_ny[o];
    const int line0 = v0 / nxo;                          // first line of the octant that the group touches
    const int nlines = (v0 + nvg - 1) / nxo - line0 + 1;

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
    const int nx = a.nx, ny = a.ny, na = a.ax_n;
    const size_t ncell = a.ncell;
    const size_t Nv = (size_t)a.Nv;
    const bool any_solid =
        a.any_solid != 0 && !(a.blk_plain != nullptr && a.blk_plain[((size_t)bzi * a.nby + byi) * a.nbx + bxi] != 0);

    auto GX = [&](int li) { return px ? x0 + li : x0 + ex - 1 - li; };
    auto GY = [&](int lj) { return py ? y0 + lj : y0 + ey - 1 - lj; };
    auto GZ = [&](int lk) { return pz ? z0 + lk : z0 + ez - 1 - lk; };
    auto CELL = [&](int x, int y, int z) { return (size_t)x + (size_t)nx * ((size_t)y + (size_t)ny * z); };

    const double *vel = static_cast<const double *>(a.vel);
    const double *mt = static_cast<const double *>(a.mtab);
    const double *coef = static_cast<const double *>(a.coef);
    const double4 *tab = static_cast<const double4 *>(a.ax_tab);
    double *FXp = static_cast<double *>(a.FX);
    double *FYp = static_cast<double *>(a.FY);
    double *FZp = static_cast<double *>(a.FZ);

    // ---- the thread's velocity ----
    const bool ok = t < nvg;
    const int vt = ok ? t : 0;
    const size_t gv = (size_t)a.oct_vstart[o] + v0 + vt;
    const int myline = (v0 + vt) / nxo - line0;
    const int xnode = (px ? a.ax_neg[0] : 0) + (v0 + vt) % nxo;
    const double axi0 = fabs(vel[gv * 4 + 0]), axi1 = fabs(vel[gv * 4 + 1]), axi2 = fabs(vel[gv * 4 + 2]);
    double ax = 0.0, ay = 0.0, az = 0.0, asum = 0.0;
    if constexpr (UNIF) {
        ax = axi0 * a.rd0[0];
        ay = axi1 * a.rd0[1];
        az = axi2 * a.rd0[2];
        asum = ax + ay + az;
    }
    const double mgx = mt[(size_t)(a.side_inflow[sidex] ? MT_INFLOW : sidex) * Nv + gv];
    const double mgy = mt[(size_t)(a.side_inflow[sidey] ? MT_INFLOW : sidey) * Nv + gv];
    // nodes of the moment phase
    for (int ix = t; ix < nxo; ix += NT) {
        const size_t g = (size_t)a.oct_vstart[o] + ix;  // the octant's first line
        xi_x[ix] = vel[g * 4];
        wxp[ix * 4] = static_cast<const double *>(a.velm)[g * 8];
    }
    const double *line_xi = vel + ((size_t)a.oct_vstart[o] + (size_t)line0 * nxo) * 4;  // first node of the first line
    for (int l = t; l < nlines; l += NT) {
        const size_t g = (size_t)a.oct_vstart[o] + (size_t)(line0 + l) * nxo;
        lw[l * LW + 9] = vel[g * 4 + 1];
        lw[l * LW] = static_cast<const double *>(a.velm)[g * 8 + 1];
    }
    auto load_centre = [&](int lk) {
        if (t < 4) cen2[lk % 2 * 4 + t] = a.centre[slice_centre(GX(0), GY(0), GZ(lk), nx, ny) + t];
    };
    // their weights about a slice's centre: warp 0 the x nodes, the others a
    // third of every line's, so that no warp runs a long chain before the sweep
    auto build_weights = [&](const double *cen) {
        const int part = t / 32, lane = t % 32;
        if (part == 0) {
            for (int ix = lane; ix < nxo; ix += 32) {
                double *e = wxp + ix * 4;
                const double x = xi_x[ix] - cen[0], wx = e[0], x2 = x * x;
                e[1] = wx * x;
                e[2] = wx * x2;
                e[3] = wx * x * x2;
            }
            return;
        }
        for (int l = lane; l < nlines; l += 32) {
            double *e = lw + l * LW;
            const double y = e[9] - cen[1], z = line_xi[(size_t)l * nxo * 4 + 2] - cen[2], W = e[0];
            if (part == 1) {
                e[1] = W * y;
                e[3] = W * y * y;
                e[5] = W * y * z;
            } else if (part == 2) {
                e[2] = W * z;
                e[4] = W * z * z;
                e[6] = W * (y * y + z * z);
            } else {
                const double Wr = W * (y * y + z * z);
                e[7] = Wr * y;
                e[8] = Wr * z;
            }
        }
    };
    load_centre(0);
    // the half of the group that this thread sums in the moment phase
    const int mcl = t % SLICE, mvp = t / SLICE;  // NT = 2 * SLICE
    const int mb = mvp * (VG / 2), me = min(mb + VG / 2, nvg);

    auto wall_rho = [&](int side, size_t cell) -> double {
        return a.side_inflow[side] ? 1.0 : a.rho_w[side * ncell + cell];
    };

    // ---- prefetch registers: halos and cell data of one slice ----
    double phx[BY], phy[BX], pc[3];
    auto prefetch = [&](int lk) {
        const int z = GZ(lk);
        {
            const int cl = t / 2, li = cl % BX, lj = cl / BX;
            if (li < ex && lj < ey) {
                const double *src = coef + CELL(GX(li), GY(lj), z) * NCOEF;
                if (t % 2 == 0) {
                    pc[0] = src[C_RTAU];
                    pc[1] = src[C_FLAGS];
                } else if (!UNIF) {
                    pc[0] = src[C_RDX];
                    pc[1] = src[C_RDY];
                    pc[2] = src[C_RDZ];
                }
            } else {
                pc[0] = 0.0;
                pc[1] = t % 2 == 0 ? flag_value<double>(F_SOLID) : 0.0;
                pc[2] = 0.0;
            }
        }
        if (xfirst) {
#pragma unroll
            for (int lj = 0; lj < BY; lj++) {
                if (lj >= ey) break;
                phx[lj] = wall_rho(sidex, CELL(GX(0), GY(lj), z)) * mgx;
            }
        } else {
            const double *fi = FXp + ((size_t)z * ny + GY(0)) * Nv + gv;
            const long long step = py ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int lj = 0; lj < BY; lj++) {
                if (lj >= ey) break;
                phx[lj] = ld_face<true>(fi + lj * step);
            }
        }
        if (yfirst) {
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
                phy[li] = wall_rho(sidey, CELL(GX(li), GY(0), z)) * mgy;
            }
        } else {
            const double *fi = FYp + ((size_t)z * nx + GX(0)) * Nv + gv;
            const long long step = px ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
                phy[li] = ld_face<true>(fi + li * step);
            }
        }
    };
    // H of every cell of slice lk and line of the group
    auto build_h = [&](int lk) {
        const size_t zc = (size_t)nx * ny * GZ(lk);
        const int yoff = a.ax_nx + (py ? a.ax_neg[1] : 0), zoff = a.ax_nx + a.ax_ny + (pz ? a.ax_neg[2] : 0);
        const int n = ey * ex * nlines;
#pragma unroll 2
        for (int e = t; e < n; e += NT) {
            const int l = e % nlines, r = e / nlines, li = r % ex, lj = r / ex;
            const double4 *rec = tab + (zc + (size_t)nx * GY(lj) + GX(li)) * na;
            const int gl = line0 + l;
            const double4 y = ld_rec(rec + yoff + gl % nyo), z = ld_rec(rec + zoff + gl / nyo);
            const double h0 = y.x * z.x, al = y.y + z.y, bl = y.z + z.z, h2 = h0 * al;
            double2 *dst = reinterpret_cast<double2 *>(H + ((size_t)(lj * BX + li) * lines_max + l) * 4);
            dst[0] = make_double2(h0, h0 * bl);
            dst[1] = make_double2(h2, h2 * bl);
        }
    };
    prefetch(0);
    build_h(0);

    // z inflow of the block: the slice starts as slice k0 - 1
    if (zfirst) {
        const double mgz = mt[(size_t)(a.side_inflow[sidez] ? MT_INFLOW : sidez) * Nv + gv];
        for (int lj = 0; lj < ey; lj++)
            for (int li = 0; li < ex; li++) {
                const double rw = wall_rho(sidez, CELL(GX(li), GY(lj), GZ(0)));
                if (ok) slice[(lj * BX + li) * CS + t] = rw * mgz;
            }
    } else {
        const long long sx = px ? (long long)Nv : -(long long)Nv;
        for (int lj = 0; lj < ey; lj++) {
            const double *fi = FZp + ((size_t)GY(lj) * nx + GX(0)) * Nv + gv;
            double v[BX];
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
                v[li] = ld_face<true>(fi + li * sx);
            }
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
                if (ok) slice[(lj * BX + li) * CS + t] = v[li];
            }
        }
    }

    const long long stepx = px ? na : -na, stepy = (py ? (long long)nx : -(long long)nx) * na;
    for (int lk = 0; lk < ez; lk++) {
        const int z = GZ(lk);
        // stage the prefetched slice data in shared memory
        if (t % 2 == 0) {
            cell4[t / 2 * 4] = pc[0];
            cflag[t / 2] = flag_bits(pc[1]);
        } else if (!UNIF) {
            cell4[t / 2 * 4 + 1] = pc[0];
            cell4[t / 2 * 4 + 2] = pc[1];
            cell4[t / 2 * 4 + 3] = pc[2];
        }
        if (ok) {
#pragma unroll
            for (int lj = 0; lj < BY; lj++) slice[(HCOL + lj) * CS + t] = phx[lj];
#pragma unroll
            for (int li = 0; li < BX; li++) slice[(HROW + li) * CS + t] = phy[li];
        }
        if (t == 0) pipe.wait(min(lk + 2, ez));
        __syncthreads();
        if (lk + 1 < ez) prefetch(lk + 1);
        // the moment phase sums about one velocity of the slice or about U^n
        const double *cen = cen2 + lk % 2 * 4;
        const bool shared_centre = cen[3] == 0.0;
        if (shared_centre) build_weights(cen);  // read after the next barrier

        // ---- sweep of the slice: Eq. (2) fused into Eq. (7), row by row ----
        // the G records of the next two cells are in flight
        const double4 *row = tab + CELL(GX(0), GY(0), z) * na + xnode;
        const int last = ex * ey - 1;
        auto g_at = [&](int n) {  // record of the n-th cell (clamped to the last)
            const int m = min(n, last), lj = m / ex, li = m - lj * ex;
            return ld_rec(row + li * stepx + lj * stepy);
        };
        double4 g1 = g_at(0), g2 = g_at(1);
        int n = 0;
        for (int lj = 0; lj < ey; lj++) {
            double fx = slice[(HCOL + lj) * CS + t];
            const double *up = slice + (lj == 0 ? HROW : (lj - 1) * BX) * CS + t;
            double *at = slice + lj * BX * CS + t;
            const double2 *h = reinterpret_cast<const double2 *>(H + ((size_t)lj * BX * lines_max + myline) * 4);
            for (int li = 0; li < ex; li++, n++) {
                const double4 g = g1;
                g1 = g2;
                g2 = g_at(n + 2);
                const double2 h01 = h[0], h23 = h[1];
                h += 2 * lines_max;
                double fy = up[li * CS], fz = at[li * CS];
                if (any_solid) {
                    const int flags = cflag[lj * BX + li];
                    if (flags & F_SOLID) continue;
                    // the x value of a cell behind a solid one is not in fx
                    fx = li > 0 ? at[(li - 1) * CS] : slice[(HCOL + lj) * CS + t];
                    const size_t cell = CELL(GX(li), GY(lj), z);
                    const double ms = mt[(size_t)MT_SOLID * Nv + gv];
                    if (flags & (F_SOLID_SIDE << sidex)) fx = a.rho_w[sidex * ncell + cell] * ms;
                    if (flags & (F_SOLID_SIDE << sidey)) fy = a.rho_w[sidey * ncell + cell] * ms;
                    if (flags & (F_SOLID_SIDE << sidez)) fz = a.rho_w[sidez * ncell + cell] * ms;
                }
                const double *c4 = cell4 + (lj * BX + li) * 4;
                double den;
                if constexpr (UNIF) {
                    den = c4[0] + asum;
                } else {
                    ax = axi0 * c4[1];
                    ay = axi1 * c4[2];
                    az = axi2 * c4[3];
                    den = c4[0] + ax + ay + az;
                }
                double num = g.x * h01.x;
                num = fma(g.y, h01.y, num);
                num = fma(g.z, h23.x, num);
                num = fma(g.w, h23.y, num);
                num = fma(az, fz, num);
                num = fma(ay, fy, num);
                num = fma(ax, fx, num);
                double r;
                asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(den));
                const double e = fma(-den, r, 1.0), q = num * r;
                fx = fma(q, fma(e, e, e), q);
                if (ok) at[li * CS] = fx;
            }
        }
        // outflow of the slice through the block's downwind x and y faces
        if (!xlast && ok) {
            double *fo = FXp + ((size_t)z * ny + GY(0)) * Nv + gv;
            const long long step = py ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int lj = 0; lj < BY; lj++) {
                if (lj >= ey) break;
                fo[lj * step] = slice[(lj * BX + ex - 1) * CS + t];
            }
        }
        if (!ylast && ok) {
            double *fo = FYp + ((size_t)z * nx + GX(0)) * Nv + gv;
            const long long step = px ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
                fo[li * step] = slice[((ey - 1) * BX + li) * CS + t];
            }
        }
        __syncthreads();
        if (t == 0) pipe.announce(lk + 1, ez);
        if (lk + 1 < ez) {
            build_h(lk + 1);
            load_centre(lk + 1);
        }

        // ---- moments of the slice about its centre over the group's velocities ----
        const int li = mcl % BX, lj = mcl / BX;
        const int flags = cflag[mcl];
        const bool live = li < ex && lj < ey && !(flags & F_SOLID);
        double S[P_FX];
#pragma unroll
        for (int q = 0; q < P_FX; q++) S[q] = 0.0;
        const double *m2u = coef + CELL(GX(li), GY(lj), z) * NCOEF + C_M2UX;  // -2 U^n, read where live
        if (live && shared_centre) {
            const double *sp = slice + mcl * CS;
            int v = mb, ix = (v0 + mb) % nxo, l = (v0 + mb) / nxo - line0;
            while (v < me) {
                // the part of line l in this half
                const int end = min(me, v + nxo - ix);
                double P0 = 0.0, P1 = 0.0, P2 = 0.0, P3 = 0.0;
                const double2 *wp = reinterpret_cast<const double2 *>(wxp) + 2 * ix;
#pragma unroll 4
                for (; v < end; v++, wp += 2) {
                    const double f = sp[v];
                    const double2 w01 = wp[0], w23 = wp[1];
                    P0 = fma(w01.x, f, P0);
                    P1 = fma(w01.y, f, P1);
                    P2 = fma(w23.x, f, P2);
                    P3 = fma(w23.y, f, P3);
                }
                const double2 *e = reinterpret_cast<const double2 *>(lw + l * LW);
                const double2 e01 = e[0], e23 = e[1], e45 = e[2], e67 = e[3];
                const double W = e01.x, Wy = e01.y, Wz = e23.x;
                S[P_S0] = fma(W, P0, S[P_S0]);
                S[P_S1X] = fma(W, P1, S[P_S1X]);
                S[P_S1Y] = fma(Wy, P0, S[P_S1Y]);
                S[P_S1Z] = fma(Wz, P0, S[P_S1Z]);
                S[P_S2XX] = fma(W, P2, S[P_S2XX]);
                S[P_S2YY] = fma(e23.y, P0, S[P_S2YY]);
                S[P_S2ZZ] = fma(e45.x, P0, S[P_S2ZZ]);
                S[P_S2XY] = fma(Wy, P1, S[P_S2XY]);
                S[P_S2XZ] = fma(Wz, P1, S[P_S2XZ]);
                S[P_S2YZ] = fma(e45.y, P0, S[P_S2YZ]);
                S[P_S3X] = fma(e67.x, P1, fma(W, P3, S[P_S3X]));
                S[P_S3Y] = fma(e67.y, P0, fma(Wy, P2, S[P_S3Y]));
                S[P_S3Z] = fma(lw[l * LW + 8], P0, fma(Wz, P2, S[P_S3Z]));
                ix = 0;
                l++;
            }
        } else if (live) {
            const double cx = -0.5 * m2u[0], cy = -0.5 * m2u[1], cz = -0.5 * m2u[2];
            const double *sp = slice + mcl * CS;
            int v = mb, ix = (v0 + mb) % nxo, l = (v0 + mb) / nxo - line0;
            while (v < me) {
                const int end = min(me, v + nxo - ix);
                double P0 = 0.0, P1 = 0.0, P2 = 0.0, P3 = 0.0;
#pragma unroll 4
                for (; v < end; v++, ix++) {
                    const double x = xi_x[ix] - cx, p0 = wxp[ix * 4] * sp[v], p1 = p0 * x, p2 = p1 * x;
                    P0 += p0;
                    P1 += p1;
                    P2 += p2;
                    P3 = fma(p2, x, P3);
                }
                const double y = lw[l * LW + 9] - cy, z2 = line_xi[(size_t)l * nxo * 4 + 2] - cz, W = lw[l * LW];
                const double r = fma(y, y, z2 * z2);
                const double q0 = W * P0, q1 = W * P1, q2 = W * P2, y0 = y * q0, z0q = z2 * q0, e2 = fma(r, q0, q2);
                S[P_S0] += q0;
                S[P_S1X] += q1;
                S[P_S1Y] += y0;
                S[P_S1Z] += z0q;
                S[P_S2XX] += q2;
                S[P_S2YY] = fma(y, y0, S[P_S2YY]);
                S[P_S2ZZ] = fma(z2, z0q, S[P_S2ZZ]);
                S[P_S2XY] = fma(y, q1, S[P_S2XY]);
                S[P_S2XZ] = fma(z2, q1, S[P_S2XZ]);
                S[P_S2YZ] = fma(z2, y0, S[P_S2YZ]);
                S[P_S3X] = fma(r, q1, fma(W, P3, S[P_S3X]));
                S[P_S3Y] = fma(y, e2, S[P_S3Y]);
                S[P_S3Z] = fma(z2, e2, S[P_S3Z]);
                ix = 0;
                l++;
            }
        }
        // combine the two halves; the incoming flux towards the wall ahead is
        // the octant's first moment along the axis (about 0) up to sign
        if (mvp == 1) {
#pragma unroll
            for (int q = 0; q < P_FX; q++) red[q * SLICE + mcl] = S[q];
        }
        __syncthreads();
        if (mvp == 0 && li < ex && lj < ey) {
#pragma unroll
            for (int q = 0; q < P_FX; q++) S[q] += red[q * SLICE + mcl];
            double out[NPART];
#pragma unroll
            for (int q = 0; q < P_FX; q++) out[q] = S[q];
            auto flux = [&](int side, bool up, int d, double s1) {
                if (!live || !(flags & (F_WALL_SIDE << side))) return 0.0;
                const double f = fma(shared_centre ? cen[d] : -0.5 * m2u[d], S[P_S0], s1);
                return up ? f : -f;
            };
            out[P_FX] = flux(headx, px, 0, S[P_S1X]);
            out[P_FY] = flux(heady, py, 1, S[P_S1Y]);
            out[P_FZ] = flux(headz, pz, 2, S[P_S1Z]);
            double2 *pp = reinterpret_cast<double2 *>(scratch + ((size_t)lk * SLICE + mcl) * NPART);
#pragma unroll
            for (int q = 0; q < NPART; q += 2) pp[q / 2] = make_double2(out[q], out[q + 1]);
        }
        // the next slice's halo row overwrites the reduction buffer
        __syncthreads();
    }

    // z outflow of the block for the next stage (own velocities only)
    if (!zlast && ok) {
        for (int lj = 0; lj < ey; lj++)
            for (int li = 0; li < ex; li++)
                FZp[((size_t)GY(lj) * nx + GX(li)) * Nv + gv] = slice[(lj * BX + li) * CS + t];
    }
}

template <bool UNIF>
__global__ void __launch_bounds__(NT, 2) sweep_d_kernel(const BatchSweepArgs b, const int lines_max)
{
    extern __shared__ __align__(16) unsigned char smem[];
    persistent_loop<double>(b, [&](const SweepArgs &a, const int4 w, const int vg, void *scratch, Pipe &pipe) {
        sweep_item_d<UNIF>(a, w, vg, smem, static_cast<double *>(scratch), pipe, lines_max);
    });
}

using Persistent = void (*)(BatchSweepArgs, int);
Persistent pick(const SweepKind &k) { return k.uniform ? sweep_d_kernel<true> : sweep_d_kernel<false>; }

}  // namespace

size_t sweep_d_smem_bytes(const SweepKind &k, int nxo_max) { return LayoutD::total(nxo_max, k.lines_max); }

int sweep_d_occupancy(const SweepKind &k, size_t smem)
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

cudaError_t launch_sweep_d(const SweepKind &k, const BatchSweepArgs &b, int nxo_max, int grid, cudaStream_t s)
{
    const size_t smem = sweep_d_smem_bytes(k, nxo_max);
    const Persistent fn = pick(k);
    const cudaError_t e = ensure_smem(reinterpret_cast<const void *>(fn), smem);
    if (e != cudaSuccess) return e;
    fn<<<grid, NT, smem, s>>>(b, k.lines_max);
    return cudaGetLastError();
}

cudaError_t launch_axis_tables(const void *coef, const double *nodes, unsigned long long ncell, int nvx, int nvy,
                               int na, void *tab, cudaStream_t s)
{
    const size_t n = (size_t)ncell * na;
    axis_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(static_cast<const double *>(coef), nodes, ncell, nvx, nvy,
                                                            na, static_cast<double4 *>(tab));
    return cudaGetLastError();
}

cudaError_t launch_slice_centres(const void *coef, int nx, int ny, int nz, double *centre, cudaStream_t s)
{
    const unsigned nb = (unsigned)((nx + BX - 1) / BX) * ((ny + BY - 1) / BY) * nz;
    centre_kernel<<<nb, SLICE, 0, s>>>(static_cast<const double *>(coef), nx, ny, centre);
    return cudaGetLastError();
}

}  // namespace kgs
