// kgs_sweep.cu -- the fused equilibrium + upwind implicit sweep + moment
// kernel of one outer iteration (arXiv 1810.00348, Eqs. (2), (5), (7), (9)).
// This is the general form: FP32 with one velocity per thread, the second
// order, FP64 without axis factors, and, with one launch per stage only, FP32
// with two velocities per thread without packed slots.  kgs_sweep_f2.cu and
// kgs_sweep_d.cu serve the first order in FP32 and FP64 otherwise.
//
// Work decomposition.  The physical grid is cut into blocks of BX x BY x bz
// cells.  For the velocities of octant o (signs of xi_x, xi_y, xi_z) a block
// depends only on its three upwind neighbour blocks, so the blocks are swept
// in diagonal stages (block coordinates reflected so that the sweep runs
// towards +x, +y, +z): stage s holds every block whose reflected coordinates
// sum to s, for all eight octants at once.  A work item is (octant, block,
// group of vg_size velocities of that octant).  The persistent kernel claims
// items in stage order and waits (bounded) for the progress of the item's
// three upwind blocks, slice by slice, so one launch covers the whole sweep; the
// kernel with one launch per stage serves the entry point that allocates no
// device memory (no flags needed).  Velocities
// are independent within an outer iteration (Eq. (6) lags f^S, tau and
// rho_w), which is what lets all octants and all velocity groups run
// concurrently.
//
// Inside a CTA each thread owns TV velocities of the group and marches the
// block slice by slice along z.  The XY slice of every velocity of the group
// lives in shared memory and is updated in place (Section 3.2: the value of
// slice k-1 at (i, j) is read once, by the update of (i, j, k), just before
// it is overwritten), with a halo row and column holding the values that
// enter the slice from the upwind neighbour blocks or the domain boundary.
// Within a slice a thread visits the cells by anti-diagonals i + j = d: the
// cells of one diagonal are independent and their upwind values (i-1, j),
// (i, j-1) were written on the previous diagonal.  Each update is the
// pointwise solution of Eq. (7):
//     f = (f^S/tau + sum_d a_d f_up,d) / (1/tau + sum_d a_d),  a_d = |xi_d|/dx_d,
// with the Shakhov equilibrium f^S of Eq. (2) computed on the fly from the
// lagged coefficients of the cell.
//
// After each slice the threads switch to a cell-per-thread layout and sum
// the slice's moments over the group's velocities: the 13 sums about the
// lagged velocity U^n and the incoming wall fluxes of Eq. (9).  Along an
// x-line of the tensor-product velocity grid only c_x changes, so a thread
// accumulates P_a = sum w_x c_x^a f (a = 0..3) and folds them with the line's
// c_y, c_z and w_y w_z at the end of the line.  In FP32 the factors c_d =
// xi_d - U_d are carried as float pairs (hi + lo, with first-order
// corrections): their rounding would otherwise repeat identically on every
// line and add up coherently in the heat flux.  The line folds go into
// Kahan-compensated sums.  The per-(group, cell) partial (FP64, or an FP32
// Kahan pair) goes to a per-CTA scratch block in the persistent kernel, which
// then adds it, in the fixed order of an accumulator chain, into one of a few
// per-cell accumulators (no atomics, no buffer that grows with the phase
// space); the staged kernel writes per-group partials for a fixed-order
// reduction kernel.  The FP32 sweep carries the deviation g = f - M_ref from
// a per-velocity reference Maxwellian, whose moments are added in FP64 when
// the sums are formed.  Block faces between stages go through three face
// planes in global memory indexed by the cell position on the face: a block
// reads the plane entries written by its upwind neighbour in the previous
// stage before overwriting them with its own outflow.
#include <map>
#include <mutex>
#include <utility>

#include "kgs_sweep_dev.cuh"

namespace kgs {

// The dynamic shared-memory limit is an attribute of a kernel on one device:
// it is raised (never lowered) on the current device before a launch that
// needs more than that device has been given, under a lock so that host
// threads launching the same kernel do not undo each other's setting.
namespace {
std::mutex g_smem_mutex;
std::map<std::pair<int, const void *>, size_t> g_smem_set;
}  // namespace

cudaError_t ensure_smem(const void *fn, size_t bytes)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(g_smem_mutex);
    size_t &have = g_smem_set[std::make_pair(dev, fn)];
    if (bytes <= have) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) have = bytes;
    return e;
}
namespace {

template <typename Real, int TV, int ORDER = 1>
struct SmemLayout {
    static constexpr int VG = NT * TV;
    static constexpr int CS = VG + 1;  // odd cell stride: conflict-free per-cell reads
    static constexpr int H = ORDER;    // halo width: the upwind cells a stencil reaches
    static constexpr int PX = BX + H;  // slice positions per row, halo included
    static constexpr size_t slice_bytes = align16(sizeof(Real) * (BY + H) * PX * CS);
    // order 2: slice k-2 at the block's own cells
    static constexpr size_t slice2_bytes = ORDER == 2 ? align16(sizeof(Real) * BY * BX * CS) : 0;
    static constexpr size_t coef_bytes = align16(sizeof(Real) * SLICE * NCOEF);
    static constexpr size_t vt_bytes = align16(sizeof(Real) * VG * VT);
    static constexpr size_t red_bytes = sizeof(double) * NPART * SLICE;
    // The halo rows of the slice (H rows of PX cell positions) are not read
    // during the moment phase, so the reduction buffer of the two velocity
    // halves lives there when it fits (it does for 256 FP32 or 128 FP64
    // velocities); a barrier at the end of the slice keeps the next slice's
    // halo from overwriting it early.
    static constexpr bool red_in_halo = sizeof(Real) * H * PX * CS >= red_bytes;
    static constexpr size_t off_coef = slice_bytes + slice2_bytes;
    static constexpr size_t off_vt = off_coef + coef_bytes;
    static constexpr size_t off_red = off_vt + vt_bytes;
    static constexpr size_t fixed = off_red + (red_in_halo ? 0 : red_bytes);
    static int cx_stride(int nxm) { return nxm | 1; }  // odd: conflict-free per-cell reads
    // line: x-lines of LINE nodes keep their c_x in registers (no c_x tables)
    static size_t total(int nxm, bool line)
    {
        return fixed + align16(sizeof(Real) * 2 * nxm) + (line ? 0 : 2 * align16(sizeof(Real) * SLICE * cx_stride(nxm)));
    }
};
// One work item: block w = (octant, reflected block coordinates) and
// velocity group vgy of that octant.  Called by every thread of the CTA.
//
// The item's moment partials go, per (group, cell), to a.part (staged sweep,
// COHERENT false) or, in the persistent sweep, to this CTA's scratch block
// [bz * SLICE][NPART] indexed by the cell's place in the block, from where
// chain_add moves them into the ordered accumulators.
//
// ORDER 2 (second-order upwind, single contexts on solid-free uniform grids):
// slice2 keeps slice k-2 at the block's cells, the halo is two cells wide,
// and FX2/FY2/FZ2 carry the block outflow one cell further upwind.
template <typename Real, int TV, int LINE, bool COHERENT, bool UNIF, int ORDER = 1, bool DEV = false>
__device__ __forceinline__ void sweep_item(const SweepArgs &a, const int4 w, const int vgy, unsigned char *smem,
                                           void *scratch, Pipe *pipe)
{
    // the deviation-form FP32 source (uniform grids: it uses the width slots)
    constexpr bool DEVF = sizeof(Real) == 4 && (ORDER == 2 || DEV);
    static_assert(!DEVF || UNIF, "the deviation-form source needs a uniform grid");
    using L = SmemLayout<Real, TV, ORDER>;
    constexpr int VG = L::VG;
    constexpr int CS = L::CS;
    constexpr int H = L::H, PX = L::PX;
    const int nxm = a.nxo_max;
    Real *slice = reinterpret_cast<Real *>(smem);
    Real *slice2 = reinterpret_cast<Real *>(smem + L::slice_bytes);  // order 2 only
    Real *cs = reinterpret_cast<Real *>(smem + L::off_coef);
    Real *vt = reinterpret_cast<Real *>(smem + L::off_vt);
    double *mred = L::red_in_halo ? reinterpret_cast<double *>(smem) : reinterpret_cast<double *>(smem + L::off_red);
    const int cxs = nxm | 1;
    Real *xn = reinterpret_cast<Real *>(smem + L::fixed);  // [nxm][2]
    Real *cxh = reinterpret_cast<Real *>(smem + L::fixed + align16(sizeof(Real) * 2 * nxm));  // [SLICE][cxs]
    Real *cxl = cxh + align16(sizeof(Real) * SLICE * cxs) / sizeof(Real);                    // [SLICE][cxs]

    const int t = threadIdx.x;
    const int o = w.x;
    const int vcount = a.oct_vcount[o];
    const int v0 = vgy * VG;
    if (v0 >= vcount) return;
    const int nvg = min(VG, vcount - v0);
    const int gvbase = a.oct_vstart[o] + v0;
    const int vgid = a.oct_vgbase[o] + vgy;
    const int nxo = a.oct_nx[o];

    // Octant bit d set: xi_d >= 0, sweep towards +d.
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
    // solid cells or solid neighbours in this block (a.blk_plain marks the
    // physical blocks that have neither; without it every block of a problem
    // with solid cells counts as having them)
    const bool any_solid =
        a.any_solid != 0 && !(a.blk_plain != nullptr && a.blk_plain[((size_t)bzi * a.nby + byi) * a.nbx + bxi] != 0);

    auto GX = [&](int li) { return px ? x0 + li : x0 + ex - 1 - li; };
    auto GY = [&](int lj) { return py ? y0 + lj : y0 + ey - 1 - lj; };
    auto GZ = [&](int lk) { return pz ? z0 + lk : z0 + ez - 1 - lk; };
    auto SL = [&](int li, int lj) { return ((lj + H) * PX + (li + H)) * CS; };  // li, lj may be -1 (-2: order 2)
    auto CELL = [&](int x, int y, int z) { return (size_t)x + (size_t)nx * ((size_t)y + (size_t)ny * z); };

    const Real *vel = static_cast<const Real *>(a.vel);
    const Real *velm = static_cast<const Real *>(a.velm);
    const Real *mt = static_cast<const Real *>(a.mtab);
    const Real *coef = static_cast<const Real *>(a.coef);
    Real *FXp = static_cast<Real *>(a.FX);
    Real *FYp = static_cast<Real *>(a.FY);
    Real *FZp = static_cast<Real *>(a.FZ);
    Real *FX2p = static_cast<Real *>(a.FX2);
    Real *FY2p = static_cast<Real *>(a.FY2);
    Real *FZ2p = static_cast<Real *>(a.FZ2);
    // order 2: index of the block's first cell along each sweep direction
    // (cells with index >= 2 have both upwind neighbours in the domain)
    const int sx0 = px ? x0 : nx - x0 - ex, sy0 = py ? y0 : ny - y0 - ey, sz0 = pz ? z0 : a.nz - z0 - ez;

    // ---- per-thread velocities (vl = t + m*NT) and the moment-phase tables ----
    // The FP32 sweep carries g = f - M_ref (mref: the reference Maxwellian of
    // the velocity); every ghost value enters as ghost - M_ref and the source
    // as f^S/tau - M_ref/tau.  The FP64 sweep carries f (mref unused).
    Real xi[TV][3], axi[TV][3], mgx[TV], mgy[TV], mgz[TV], msol[TV], mref[TV];
    Real dmref[TV];  // deviation-form source: the rounding error of M_ref
    size_t gv[TV];
    bool ok[TV];
    const int rowx = a.side_inflow[sidex] ? MT_INFLOW : sidex;
    const int rowy = a.side_inflow[sidey] ? MT_INFLOW : sidey;
    const int rowz = a.side_inflow[sidez] ? MT_INFLOW : sidez;
#pragma unroll
    for (int m = 0; m < TV; m++) {
        const int vl = t + m * NT;
        ok[m] = vl < nvg;
        gv[m] = (size_t)gvbase + (ok[m] ? vl : 0);
        xi[m][0] = vel[gv[m] * 4 + 0];
        xi[m][1] = vel[gv[m] * 4 + 1];
        xi[m][2] = vel[gv[m] * 4 + 2];
        axi[m][0] = fabs(xi[m][0]);
        axi[m][1] = fabs(xi[m][1]);
        axi[m][2] = fabs(xi[m][2]);
        // x-line factor w_x; line data for the fold: xi_y, xi_z (hi, lo), w_y w_z
        Real *e = vt + vl * VT;
        e[0] = ok[m] ? velm[gv[m] * 8 + 0] : Real(0);
        e[1] = xi[m][1];
        e[2] = xi[m][2];
        e[3] = ok[m] ? velm[gv[m] * 8 + 1] : Real(0);
        e[4] = velm[gv[m] * 8 + 3];
        e[5] = velm[gv[m] * 8 + 4];
        e[6] = Real(0);
        e[7] = Real(0);
        mgx[m] = mt[(size_t)rowx * Nv + gv[m]];
        mgy[m] = mt[(size_t)rowy * Nv + gv[m]];
        mgz[m] = mt[(size_t)rowz * Nv + gv[m]];
        msol[m] = mt[(size_t)MT_SOLID * Nv + gv[m]];
        mref[m] = sizeof(Real) == 4 ? velm[gv[m] * 8 + 5] : Real(0);
        if constexpr (DEVF) dmref[m] = velm[gv[m] * 8 + 6];
    }
    // ghost value rho_w * (unit wall or free-stream Maxwellian), as carried
    auto ghost = [&](Real rw, Real mg, int m) -> Real {
        if constexpr (sizeof(Real) == 4)
            return fma(rw, mg, -mref[m]);
        else
            return rw * mg;
    };
    // |xi|^2 of each velocity, rounded once from its FP64 value
    Real xsq[TV];
#pragma unroll
    for (int m = 0; m < TV; m++) {
        const double x0 = xi[m][0], x1 = xi[m][1], x2 = xi[m][2];
        xsq[m] = Real(x0 * x0 + x1 * x1 + x2 * x2);
    }
    // uniform grid: the upwind coefficients a_d = abs(xi_d) / dx_d and their
    // sum depend on the velocity only
    Real adx[TV][3], asum[TV];
#pragma unroll
    for (int m = 0; m < TV; m++) {
        if constexpr (UNIF) {
            adx[m][0] = axi[m][0] * Real(a.rd0[0]);
            adx[m][1] = axi[m][1] * Real(a.rd0[1]);
            adx[m][2] = axi[m][2] * Real(a.rd0[2]);
            asum[m] = adx[m][0] + adx[m][1] + adx[m][2];
        } else {
            adx[m][0] = adx[m][1] = adx[m][2] = asum[m] = Real(0);
        }
    }
    // x nodes of the octant in line order (the first nxo velocities of the octant)
    for (int ix = t; ix < nxo; ix += NT) {
        const size_t g = (size_t)a.oct_vstart[o] + ix;
        xn[ix * 2 + 0] = vel[g * 4 + 0];
        xn[ix * 2 + 1] = velm[g * 8 + 2];
    }

    // Ghost value entering through domain side `side` at cell `cell`:
    // free stream, or rho_w times the unit wall Maxwellian (Eq. (8)).
    auto wall_rho = [&](int side, size_t cell) -> Real {
        return a.side_inflow[side] ? Real(1) : Real(a.rho_w[side * ncell + cell]);
    };

    // ---- prefetch registers: coefficients and halos of one slice ----
    Real pc[CPF];
    Real phx[BY][TV], phy[BX][TV];
    Real phx2[ORDER == 2 ? BY : 1][TV], phy2[ORDER == 2 ? BX : 1][TV];  // order 2: second halo column / row
    auto prefetch = [&](int lk) {
        const int z = GZ(lk);
        const int cl = (t * CPF) / NCOEF, q0 = (t * CPF) % NCOEF;
        const int li = cl % BX, lj = cl / BX;
        if (li < ex && lj < ey) {
            const Real *src = coef + CELL(GX(li), GY(lj), z) * NCOEF + q0;
#pragma unroll
            for (int q = 0; q < CPF; q++) pc[q] = src[q];
        } else {
#pragma unroll
            for (int q = 0; q < CPF; q++) pc[q] = (q0 + q == C_FLAGS) ? flag_value<Real>(F_SOLID) : Real(0);
        }
        if (xfirst) {
#pragma unroll
            for (int lj2 = 0; lj2 < BY; lj2++) {
                if (lj2 >= ey) break;
                const Real rw = wall_rho(sidex, CELL(GX(0), GY(lj2), z));
#pragma unroll
                for (int m = 0; m < TV; m++) phx[lj2][m] = ghost(rw, mgx[m], m);
            }
        } else {
            const Real *fi = FXp + ((size_t)z * ny + GY(0)) * Nv;
            const long long step = py ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int lj2 = 0; lj2 < BY; lj2++) {
                if (lj2 >= ey) break;
#pragma unroll
                for (int m = 0; m < TV; m++)
                    phx[lj2][m] = ok[m] ? ld_face<COHERENT>(fi + lj2 * step + (long long)gv[m]) : Real(0);
            }
            if constexpr (ORDER == 2) {
                const Real *fi2 = FX2p + ((size_t)z * ny + GY(0)) * Nv;
#pragma unroll
                for (int lj2 = 0; lj2 < BY; lj2++) {
                    if (lj2 >= ey) break;
#pragma unroll
                    for (int m = 0; m < TV; m++)
                        phx2[lj2][m] = ok[m] ? ld_face<COHERENT>(fi2 + lj2 * step + (long long)gv[m]) : Real(0);
                }
            }
        }
        if (yfirst) {
#pragma unroll
            for (int li2 = 0; li2 < BX; li2++) {
                if (li2 >= ex) break;
                const Real rw = wall_rho(sidey, CELL(GX(li2), GY(0), z));
#pragma unroll
                for (int m = 0; m < TV; m++) phy[li2][m] = ghost(rw, mgy[m], m);
            }
        } else {
            const Real *fi = FYp + ((size_t)z * nx + GX(0)) * Nv;
            const long long step = px ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int li2 = 0; li2 < BX; li2++) {
                if (li2 >= ex) break;
#pragma unroll
                for (int m = 0; m < TV; m++)
                    phy[li2][m] = ok[m] ? ld_face<COHERENT>(fi + li2 * step + (long long)gv[m]) : Real(0);
            }
            if constexpr (ORDER == 2) {
                const Real *fi2 = FY2p + ((size_t)z * nx + GX(0)) * Nv;
#pragma unroll
                for (int li2 = 0; li2 < BX; li2++) {
                    if (li2 >= ex) break;
#pragma unroll
                    for (int m = 0; m < TV; m++)
                        phy2[li2][m] = ok[m] ? ld_face<COHERENT>(fi2 + li2 * step + (long long)gv[m]) : Real(0);
                }
            }
        }
    };
    prefetch(0);

    // z inflow of the block: the slice interior starts as slice k0-1.  A row
    // of cells is loaded before it is stored, so a row's loads are in flight
    // together.
    if (zfirst) {
        for (int lj = 0; lj < ey; lj++)
            for (int li = 0; li < ex; li++) {
                const Real rw = wall_rho(sidez, CELL(GX(li), GY(lj), GZ(0)));
#pragma unroll
                for (int m = 0; m < TV; m++)
                    if (ok[m]) slice[SL(li, lj) + t + m * NT] = ghost(rw, mgz[m], m);
            }
    } else {
        const long long sx = px ? (long long)Nv : -(long long)Nv;
        for (int lj = 0; lj < ey; lj++) {
            const Real *fi = FZp + ((size_t)GY(lj) * nx + GX(0)) * Nv;
            Real v[BX][TV];
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
#pragma unroll
                for (int m = 0; m < TV; m++)
                    v[li][m] = ok[m] ? ld_face<COHERENT>(fi + li * sx + (long long)gv[m]) : Real(0);
            }
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
#pragma unroll
                for (int m = 0; m < TV; m++)
                    if (ok[m]) slice[SL(li, lj) + t + m * NT] = v[li][m];
            }
            if constexpr (ORDER == 2) {
                // slice k0-2 (the upwind block's second-last slice)
                const Real *fi2 = FZ2p + ((size_t)GY(lj) * nx + GX(0)) * Nv;
#pragma unroll
                for (int li = 0; li < BX; li++) {
                    if (li >= ex) break;
#pragma unroll
                    for (int m = 0; m < TV; m++)
                        v[li][m] = ok[m] ? ld_face<COHERENT>(fi2 + li * sx + (long long)gv[m]) : Real(0);
                }
#pragma unroll
                for (int li = 0; li < BX; li++) {
                    if (li >= ex) break;
#pragma unroll
                    for (int m = 0; m < TV; m++)
                        if (ok[m]) slice2[(lj * BX + li) * CS + t + m * NT] = v[li][m];
                }
            }
        }
    }


    for (int lk = 0; lk < ez; lk++) {
        const int z = GZ(lk);
        // stage the prefetched slice data in shared memory
#pragma unroll
        for (int q = 0; q < CPF; q++) cs[t * CPF + q] = pc[q];
#pragma unroll
        for (int lj = 0; lj < BY; lj++) {
            if (lj >= ey) break;
#pragma unroll
            for (int m = 0; m < TV; m++)
                if (ok[m]) slice[SL(-1, lj) + t + m * NT] = phx[lj][m];
        }
#pragma unroll
        for (int li = 0; li < BX; li++) {
            if (li >= ex) break;
#pragma unroll
            for (int m = 0; m < TV; m++)
                if (ok[m]) slice[SL(li, -1) + t + m * NT] = phy[li][m];
        }
        if constexpr (ORDER == 2) {
            // the second halo column / row (read only by cells with both
            // upwind neighbours in the domain, so not in a first block)
            if (!xfirst) {
#pragma unroll
                for (int lj = 0; lj < BY; lj++) {
                    if (lj >= ey) break;
#pragma unroll
                    for (int m = 0; m < TV; m++)
                        if (ok[m]) slice[SL(-2, lj) + t + m * NT] = phx2[lj][m];
                }
            }
            if (!yfirst) {
#pragma unroll
                for (int li = 0; li < BX; li++) {
                    if (li >= ex) break;
#pragma unroll
                    for (int m = 0; m < TV; m++)
                        if (ok[m]) slice[SL(li, -2) + t + m * NT] = phy2[li][m];
                }
            }
        }
        if (COHERENT && t == 0) pipe->wait(min(lk + 2, ez));
        __syncthreads();
        // c_x = xi_x - U_x of each cell of the slice as a float pair, per x node
        // (lines of LINE nodes keep theirs in registers instead)
        if constexpr (LINE == 0) {
            const int cl = t % SLICE, vp = t / SLICE;
            const Real ux = Real(-0.5) * cs[cl * NCOEF + C_M2UX];
            for (int ix = vp; ix < nxo; ix += NT / SLICE) {
                Real s, e;
                two_diff(xn[ix * 2], ux, s, e);
                cxh[cl * cxs + ix] = s;
                cxl[cl * cxs + ix] = e + xn[ix * 2 + 1];
            }
        }
        if (lk + 1 < ez) prefetch(lk + 1);

        // ---- sweep of the slice: Eq. (2) fused into Eq. (7), by anti-diagonals ----
        // FP32 deviation-form source (DEVF: order 2, or the dev_source
        // option): rtau (f^S - M_ref) evaluated as rtau M_ref (2^D shak - 1)
        // with D = log2(f^S_M / M_ref) built from per-cell terms that are small
        // near the reference state (coefficient slots C_RDX, C_RDY of uniform
        // grids), so that its rounding scales with the deviation g rather than
        // with f; the reference M_ref is the rest state and its own FP32
        // rounding error dmref is added back.
        auto dev_source = [&](const Quad<Real> &c0, const Quad<Real> &c1, const Quad<Real> &c2v,
                              const Quad<Real> &c3, int m, Real cq) -> Real {
            const Real dn = c2v.w, K = c3.x;
            const Real sd = fma(xi[m][0], c0.x, fma(xi[m][1], c0.y, xi[m][2] * c0.z));  // -2 U.xi
            const Real D = fma(xsq[m], dn, fma(sd, c1.x, K));
            const Real shm1 = cq * fma(xsq[m] + sd, c1.y, c3.z);  // Shakhov factor - 1
            const Real em = exp2m1(D);
            const Real X = fma(em, shm1, em + shm1);  // 2^D shak - 1
            return c1.z * fma(mref[m], X, dmref[m]);
        };
        // Eq. (2) fused into Eq. (7) for one cell of the slice (coefficients
        // c0..c3) and thread velocity m, from its three upwind values.
        auto cell_update = [&](const Quad<Real> &c0, const Quad<Real> &c1, const Quad<Real> &c2v,
                               const Quad<Real> &c3, int m, Real fx, Real fy, Real fz) -> Real {
          if constexpr (DEVF) {
            // uniform grids only (a_d per velocity); the update about the
            // upwind x value as below, with the deviation-form source
            const Real cq = fma(xi[m][0], c2v.x, fma(xi[m][1], c2v.y, fma(xi[m][2], c2v.z, c3.w)));
            const Real dsrc = dev_source(c0, c1, c2v, c3, m, cq);
            Real t = fma(-c1.z, fx, dsrc);
            t = fma(adx[m][1], fy - fx, t);
            t = fma(adx[m][2], fz - fx, t);
            return fma(t, rcp_approx(c1.z + asum[m]), fx);
          } else {
            const Real m2ux = c0.x, m2uy = c0.y, m2uz = c0.z, kappa = c0.w;
            const Real nexp = c1.x, rt1 = c1.y, rtau = c1.z;
            const Real qx = c2v.x, qy = c2v.y, qz = c2v.z, rdx = c2v.w;
            const Real rdy = c3.x, rdz = c3.y, shk0 = c3.z, muq = c3.w;
            // |c|^2 - |U|^2 = |xi|^2 - 2 U.xi and c.q' = xi.q' - U.q'
            const Real s = fma(xi[m][0], m2ux, fma(xi[m][1], m2uy, fma(xi[m][2], m2uz, xsq[m])));
            const Real cq = fma(xi[m][0], qx, fma(xi[m][1], qy, fma(xi[m][2], qz, muq)));
            const Real shak = fma(cq, fma(s, rt1, shk0), Real(1));
            Real src;
            if constexpr (sizeof(Real) == 4)  // kappa enters as log2(kappa) in the exponent
                src = eq_exp(fma(s, nexp, kappa)) * shak;
            else
                src = kappa * eq_exp(s * nexp) * shak;
            Real ax, ay, az, den;
            if constexpr (UNIF) {
                ax = adx[m][0];
                ay = adx[m][1];
                az = adx[m][2];
                den = rtau + asum[m];
            } else {
                ax = axi[m][0] * rdx;
                ay = axi[m][1] * rdy;
                az = axi[m][2] * rdz;
                den = rtau + ax + ay + az;
            }
            if constexpr (sizeof(Real) == 4) {
                // The same solution of Eq. (7) written about the upwind x value:
                //   f = f_x + (src - f_x/tau + a_y (f_y - f_x) + a_z (f_z - f_x)) / den.
                // On a smooth field the increment is small, so the one rounding
                // that matters is the final addition, which is unbiased.  The
                // plain form num * (1/den) scales f by the same rounding error of
                // 1/den in every cell of a velocity's characteristic, and that
                // error adds up along the sweep.
                (void)ax;
                Real t = fma(-rtau, fx + mref[m], src);
                t = fma(ay, fy - fx, t);
                t = fma(az, fz - fx, t);
                return fma(t, rcp_approx(den), fx);
            } else {
                return implicit_div(src + ax * fx + ay * fy + az * fz, den);
            }
          }
        };
        // Order 2: the three-point backward difference along an axis is
        //   a (3 f - 4 f_1 + f_2) / 2 = (3a/2) (f - h),  h = f_1 + (f_1 - f_2)/3,
        // so the update is that of Eq. (7) with the coefficient 3a/2 and the
        // extrapolated upwind value h on the axes where it applies (o2d).
        auto cell_update2 = [&](const Quad<Real> &c0, const Quad<Real> &c1, const Quad<Real> &c2v,
                                const Quad<Real> &c3, int m, Real hx, Real hy, Real hz, bool o2x, bool o2y,
                                bool o2z) -> Real {
            const Real m2ux = c0.x, m2uy = c0.y, m2uz = c0.z, kappa = c0.w;
            const Real nexp = c1.x, rt1 = c1.y, rtau = c1.z;
            const Real qx = c2v.x, qy = c2v.y, qz = c2v.z;
            const Real shk0 = c3.z, muq = c3.w;
            const Real cq = fma(xi[m][0], qx, fma(xi[m][1], qy, fma(xi[m][2], qz, muq)));
            // FP32: the deviation-form source; FP64: rtau f^S as in Eq. (7)
            Real dsrc;
            if constexpr (sizeof(Real) == 4) {
                dsrc = dev_source(c0, c1, c2v, c3, m, cq);
                (void)kappa;
            } else {
                const Real s = fma(xi[m][0], m2ux, fma(xi[m][1], m2uy, fma(xi[m][2], m2uz, xsq[m])));
                const Real shak = fma(cq, fma(s, rt1, shk0), Real(1));
                dsrc = kappa * eq_exp(s * nexp) * shak;
            }
            // uniform grids only: a_d per velocity
            const Real ax = o2x ? Real(1.5) * adx[m][0] : adx[m][0];
            const Real ay = o2y ? Real(1.5) * adx[m][1] : adx[m][1];
            const Real az = o2z ? Real(1.5) * adx[m][2] : adx[m][2];
            const Real den = rtau + ax + ay + az;
            if constexpr (sizeof(Real) == 4) {
                // about the upwind x value, as the first-order FP32 update
                Real t = fma(-rtau, hx, dsrc);
                t = fma(ay, hy - hx, t);
                t = fma(az, hz - hx, t);
                return fma(t, rcp_approx(den), hx);
            } else {
                return implicit_div(dsrc + ax * hx + ay * hy + az * hz, den);
            }
        };
        if constexpr (ORDER == 2) {
            // Generic diagonal loop with the second-order stencil.  The z
            // values of (i, j) are slice k-1 (in place) and k-2 (slice2);
            // once the cell is updated, its k-1 value moves to slice2.
            const int szk = sz0 + lk;
            const bool o2z = szk >= 2;
            const Real third = Real(1) / Real(3);
            for (int d = 0; d < ex + ey - 1; d++) {
                const int jhi = min(ey - 1, d), jlo = max(0, d - (ex - 1));
#pragma unroll
                for (int k = 0; k < BY; k++) {
                    const int lj = jhi - k;
                    if (lj >= jlo) {
                        const int li = d - lj;
                        const Real *c = cs + (lj * BX + li) * NCOEF;
                        const Quad<Real> c0 = load_quad(c), c1 = load_quad(c + 4), c2v = load_quad(c + 8),
                                         c3 = load_quad(c + 12);
                        const bool o2x = sx0 + li >= 2, o2y = sy0 + lj >= 2;
                        const int sidx = SL(li, lj), bidx = (lj * BX + li) * CS;
#pragma unroll
                        for (int m = 0; m < TV; m++) {
                            const int vl = t + m * NT;
                            const Real fz = slice[sidx + vl];
                            const Real fy = slice[sidx - PX * CS + vl];
                            const Real fx = slice[sidx - CS + vl];
                            const Real hx = o2x ? fma(fx - slice[sidx - 2 * CS + vl], third, fx) : fx;
                            const Real hy = o2y ? fma(fy - slice[sidx - 2 * PX * CS + vl], third, fy) : fy;
                            const Real hz = o2z ? fma(fz - slice2[bidx + vl], third, fz) : fz;
                            const Real f = cell_update2(c0, c1, c2v, c3, m, hx, hy, hz, o2x, o2y, o2z);
                            if (ok[m]) {
                                slice2[bidx + vl] = fz;
                                slice[sidx + vl] = f;
                            }
                        }
                    }
                }
            }
        } else if (ex == BX && ey == BY && !any_solid) {
            // Full block without solid cells: the 15 diagonals unrolled.  The
            // upwind x and y values of a cell were computed on the previous
            // diagonal by this thread and stay in registers (prev[row]); only
            // the z value (the cell itself in slice k-1) and the halo row and
            // column come from shared memory.  Every index is a compile-time
            // constant, so the cells of a diagonal form straight-line code whose
            // update chains the compiler can interleave, and a diagonal waits
            // only for register results of the one before.
            Real prev[BY][TV];
#pragma unroll
            for (int d = 0; d < BX + BY - 1; d++) {
#pragma unroll
                for (int k = 0; k < BY; k++) {
                    const int lj = (d < BY - 1 ? d : BY - 1) - k;
                    const int li = d - lj;
                    if (lj >= 0 && li < BX) {
                        const Real *c = cs + (lj * BX + li) * NCOEF;
                        const Quad<Real> c0 = load_quad(c), c1 = load_quad(c + 4), c2v = load_quad(c + 8),
                                         c3 = load_quad(c + 12);
                        const int sidx = SL(li, lj);
#pragma unroll
                        for (int m = 0; m < TV; m++) {
                            const int vl = t + m * NT;
                            const Real fz = slice[sidx + vl];
                            const Real fx = li == 0 ? slice[sidx - CS + vl] : prev[lj][m];
                            const Real fy = lj == 0 ? slice[sidx - PX * CS + vl] : prev[lj > 0 ? lj - 1 : 0][m];
                            const Real f = cell_update(c0, c1, c2v, c3, m, fx, fy, fz);
                            prev[lj][m] = f;
                            if (ok[m]) slice[sidx + vl] = f;
                        }
                    }
                }
            }
        } else {
        // The upwind values of cell (i, j) are read from the in-place slice:
        // (i-1, j) and (i, j-1) were updated on the previous diagonal, (i, j)
        // itself still holds slice k-1.  The cells of one diagonal are
        // independent, which gives up to BY update chains in flight.
        for (int d = 0; d < ex + ey - 1; d++) {
            const int jhi = min(ey - 1, d), jlo = max(0, d - (ex - 1));
#pragma unroll
            for (int k = 0; k < BY; k++) {
                const int lj = jhi - k;
                if (lj >= jlo) {
                    const int li = d - lj;
                    const Real *c = cs + (lj * BX + li) * NCOEF;
                    const Quad<Real> c0 = load_quad(c), c1 = load_quad(c + 4), c2v = load_quad(c + 8),
                                     c3 = load_quad(c + 12);
                    const int flags = flag_bits(c1.w);
                    if (!(flags & F_SOLID)) {
                        bool sol_x = false, sol_y = false, sol_z = false;
                        Real rwx = 0, rwy = 0, rwz = 0;
                        if (any_solid) {
                            const size_t cell = CELL(GX(li), GY(lj), z);
                            sol_x = flags & (F_SOLID_SIDE << sidex);
                            sol_y = flags & (F_SOLID_SIDE << sidey);
                            sol_z = flags & (F_SOLID_SIDE << sidez);
                            if (sol_x) rwx = Real(a.rho_w[sidex * ncell + cell]);
                            if (sol_y) rwy = Real(a.rho_w[sidey * ncell + cell]);
                            if (sol_z) rwz = Real(a.rho_w[sidez * ncell + cell]);
                        }
                        const int sidx = SL(li, lj);
#pragma unroll
                        for (int m = 0; m < TV; m++) {
                            const int vl = t + m * NT;
                            Real fz = slice[sidx + vl];
                            Real fy = slice[sidx - PX * CS + vl];
                            Real fx = slice[sidx - CS + vl];
                            if (any_solid) {
                                if (sol_x) fx = ghost(rwx, msol[m], m);
                                if (sol_y) fy = ghost(rwy, msol[m], m);
                                if (sol_z) fz = ghost(rwz, msol[m], m);
                            }
                            const Real f = cell_update(c0, c1, c2v, c3, m, fx, fy, fz);
                            if (ok[m]) slice[sidx + vl] = f;
                        }
                    }
                }
            }
        }
        }
        // outflow of the slice through the block's downwind x and y faces, for
        // the neighbouring blocks (own velocities, read back from the slice)
        if (!xlast) {
            Real *fo = FXp + ((size_t)z * ny + GY(0)) * Nv;
            const long long step = py ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int lj = 0; lj < BY; lj++) {
                if (lj >= ey) break;
                const Real *src = slice + SL(ex - 1, lj) + t;
#pragma unroll
                for (int m = 0; m < TV; m++)
                    if (ok[m]) fo[lj * step + (long long)gv[m]] = src[m * NT];
            }
            if constexpr (ORDER == 2) {
                // the column before the last: the halo column when ex == 1
                Real *fo2 = FX2p + ((size_t)z * ny + GY(0)) * Nv;
#pragma unroll
                for (int lj = 0; lj < BY; lj++) {
                    if (lj >= ey) break;
                    const Real *src = slice + SL(ex - 2, lj) + t;
#pragma unroll
                    for (int m = 0; m < TV; m++)
                        if (ok[m]) fo2[lj * step + (long long)gv[m]] = src[m * NT];
                }
            }
        }
        if (!ylast) {
            Real *fo = FYp + ((size_t)z * nx + GX(0)) * Nv;
            const long long step = px ? (long long)Nv : -(long long)Nv;
#pragma unroll
            for (int li = 0; li < BX; li++) {
                if (li >= ex) break;
                const Real *src = slice + SL(li, ey - 1) + t;
#pragma unroll
                for (int m = 0; m < TV; m++)
                    if (ok[m]) fo[li * step + (long long)gv[m]] = src[m * NT];
            }
            if constexpr (ORDER == 2) {
                Real *fo2 = FY2p + ((size_t)z * nx + GX(0)) * Nv;
#pragma unroll
                for (int li = 0; li < BX; li++) {
                    if (li >= ex) break;
                    const Real *src = slice + SL(li, ey - 2) + t;
#pragma unroll
                    for (int m = 0; m < TV; m++)
                        if (ok[m]) fo2[li * step + (long long)gv[m]] = src[m * NT];
                }
            }
        }
        __syncthreads();
        if (COHERENT && t == 0) pipe->announce(lk + 1, ez);

        // ---- moments of the slice over the group's velocities ----
        {
            const int cl = t % SLICE, vp = t / SLICE;  // NT = 2 * SLICE: two velocity halves
            const int li = cl % BX, lj = cl / BX;
            const bool valid = li < ex && lj < ey;
            const Real *c = cs + cl * NCOEF;
            const int flags = flag_bits(c[C_FLAGS + 0]);
            RunSum<Real> S[NPART];
            if (valid && !(flags & F_SOLID)) {
                const Real ux = Real(-0.5) * c[C_M2UX], uy = Real(-0.5) * c[C_M2UY], uz = Real(-0.5) * c[C_M2UZ];
                const bool wx = flags & (F_WALL_SIDE << headx);
                const bool wy = flags & (F_WALL_SIDE << heady);
                const bool wz = flags & (F_WALL_SIDE << headz);
                const Real sgnx = px ? Real(1) : Real(-1);
                const Real *sp = slice + SL(li, lj);
                const int vbeg = vp * (VG / 2);
                const int vend = min(vbeg + VG / 2, nvg);
                // fold the line sums P_a (x-line of the tensor-product grid ending at
                // velocity ve-1) with the line's c_y, c_z and w_y w_z
                if constexpr (sizeof(Real) == 4) {
                    // fold the line sums P_a (x-line of the tensor-product grid ending at
                    // velocity ve-1) with the line's c_y, c_z and w_y w_z
                    auto fold = [&](Real P0, Real P1, Real P2, Real P3, int ve) {
                        const Real *e = vt + (ve - 1) * VT;
                        Real cy, cyl, cz, czl;
                        two_diff(e[1], uy, cy, cyl);
                        two_diff(e[2], uz, cz, czl);
                        cyl += e[4];
                        czl += e[5];
                        const Real W = e[3];
                        const Real q0 = W * P0, q1 = W * P1, q2 = W * P2;
                        const Real r2 = fma(cy, cy, cz * cz);
                        const Real r2l = Real(2) * fma(cy, cyl, cz * czl);
                        S[P_S0].add(q0);
                        S[P_S1X].add(q1);
                        S[P_S1Y].add(fma(cy, q0, cyl * q0));
                        S[P_S1Z].add(fma(cz, q0, czl * q0));
                        S[P_S2XX].add(q2);
                        S[P_S2YY].add(fma(cy, cy, Real(2) * cy * cyl) * q0);
                        S[P_S2ZZ].add(fma(cz, cz, Real(2) * cz * czl) * q0);
                        S[P_S2XY].add(fma(cy, q1, cyl * q1));
                        S[P_S2XZ].add(fma(cz, q1, czl * q1));
                        S[P_S2YZ].add(fma(cy, cz, fma(cyl, cz, cy * czl)) * q0);
                        S[P_S3X].add(fma(W, P3, fma(r2, q1, r2l * q1)));
                        const Real e2 = fma(r2, q0, fma(r2l, q0, q2));
                        S[P_S3Y].add(fma(cy, e2, cyl * e2));
                        S[P_S3Z].add(fma(cz, e2, czl * e2));
                        // incoming flux w |xi_d| f towards the wall ahead
                        if (wx) S[P_FX].add(sgnx * fma(ux, q0, q1));
                        if (wy) S[P_FY].add(fabs(e[1]) * q0);
                        if (wz) S[P_FZ].add(fabs(e[2]) * q0);
                    };
                    if constexpr (LINE > 0) {
                        // Every x-line has LINE nodes and the thread's range holds whole
                        // lines: the c_x pairs and w_x of the LINE nodes stay in registers.
                        Real cxr[LINE], cxlr[LINE], wxr[LINE];
    #pragma unroll
                        for (int ix = 0; ix < LINE; ix++) {
                            Real hi, lo;
                            two_diff(xn[ix * 2], ux, hi, lo);
                            cxr[ix] = hi;
                            cxlr[ix] = lo + xn[ix * 2 + 1];
                            wxr[ix] = vt[(vbeg + ix) * VT];
                        }
                        for (int v = vbeg; v < vend; v += LINE) {
                            Real P0 = 0, P1 = 0, P2 = 0, P3 = 0, C1 = 0, C2 = 0, C3 = 0;
    #pragma unroll
                            for (int ix = 0; ix < LINE; ix++) {
                                const Real f = sp[v + ix];
                                const Real cx = cxr[ix];
                                const Real t0 = wxr[ix] * f;
                                const Real t1 = t0 * cx;
                                const Real t2 = t1 * cx;
                                P0 += t0;
                                P1 += t1;
                                P2 += t2;
                                P3 = fma(t2, cx, P3);
                                C1 = fma(t0, cxlr[ix], C1);
                                C2 = fma(t1, cxlr[ix], C2);
                                C3 = fma(t2, cxlr[ix], C3);
                            }
                            // first-order corrections for the low part of c_x
                            fold(P0, P1 + C1, fma(Real(2), C2, P2), fma(Real(3), C3, P3), v + LINE);
                        }
                    } else {
                        const Real *cxhc = cxh + cl * cxs, *cxlc = cxl + cl * cxs;
                        int v = vbeg;
                        while (v < vend) {
                            // one x-line segment [v, ve): velocities with the same (xi_y, xi_z)
                            const int ix0 = (v0 + v) % nxo;
                            const int ve = min(vend, v + (nxo - ix0));
                            Real P0 = 0, P1 = 0, P2 = 0, P3 = 0, C1 = 0, C2 = 0, C3 = 0;
    #pragma unroll 4
                            for (int vv = v; vv < ve; vv++) {
                                const int ix = ix0 + (vv - v);
                                const Real f = sp[vv];
                                const Real cx = cxhc[ix], cxlo = cxlc[ix];
                                const Real t0 = vt[vv * VT] * f;
                                const Real t1 = t0 * cx;
                                const Real t2 = t1 * cx;
                                P0 += t0;
                                P1 += t1;
                                P2 += t2;
                                P3 = fma(t2, cx, P3);
                                C1 = fma(t0, cxlo, C1);
                                C2 = fma(t1, cxlo, C2);
                                C3 = fma(t2, cxlo, C3);
                            }
                            fold(P0, P1 + C1, fma(Real(2), C2, P2), fma(Real(3), C3, P3), ve);
                            v = ve;
                        }
                    }
                } else {
                    // FP64: the rounding of c = xi - U^n is far below the path's
                    // tolerance, so the float-pair corrections of the FP32 path are
                    // left out (fewer operations and registers).
                    auto fold = [&](Real P0, Real P1, Real P2, Real P3, int ve) {
                        const Real *e = vt + (ve - 1) * VT;
                        const Real cy = e[1] - uy, cz = e[2] - uz;
                        const Real W = e[3];
                        const Real q0 = W * P0, q1 = W * P1, q2 = W * P2;
                        const Real r2 = fma(cy, cy, cz * cz);
                        S[P_S0].add(q0);
                        S[P_S1X].add(q1);
                        S[P_S1Y].add(cy * q0);
                        S[P_S1Z].add(cz * q0);
                        S[P_S2XX].add(q2);
                        S[P_S2YY].add(cy * cy * q0);
                        S[P_S2ZZ].add(cz * cz * q0);
                        S[P_S2XY].add(cy * q1);
                        S[P_S2XZ].add(cz * q1);
                        S[P_S2YZ].add(cy * cz * q0);
                        S[P_S3X].add(fma(W, P3, r2 * q1));
                        const Real e2 = fma(r2, q0, q2);
                        S[P_S3Y].add(cy * e2);
                        S[P_S3Z].add(cz * e2);
                        if (wx) S[P_FX].add(sgnx * fma(ux, q0, q1));
                        if (wy) S[P_FY].add(fabs(e[1]) * q0);
                        if (wz) S[P_FZ].add(fabs(e[2]) * q0);
                    };
                    if constexpr (LINE > 0) {
                        Real cxr[LINE], wxr[LINE];
    #pragma unroll
                        for (int ix = 0; ix < LINE; ix++) {
                            cxr[ix] = xn[ix * 2] - ux;
                            wxr[ix] = vt[(vbeg + ix) * VT];
                        }
                        for (int v = vbeg; v < vend; v += LINE) {
                            Real P0 = 0, P1 = 0, P2 = 0, P3 = 0;
    #pragma unroll
                            for (int ix = 0; ix < LINE; ix++) {
                                const Real f = sp[v + ix];
                                const Real cx = cxr[ix];
                                const Real t0 = wxr[ix] * f;
                                const Real t1 = t0 * cx;
                                const Real t2 = t1 * cx;
                                P0 += t0;
                                P1 += t1;
                                P2 += t2;
                                P3 = fma(t2, cx, P3);
                            }
                            fold(P0, P1, P2, P3, v + LINE);
                        }
                    } else {
                        const Real *cxhc = cxh + cl * cxs;
                        int v = vbeg;
                        while (v < vend) {
                            const int ix0 = (v0 + v) % nxo;
                            const int ve = min(vend, v + (nxo - ix0));
                            Real P0 = 0, P1 = 0, P2 = 0, P3 = 0;
    #pragma unroll 4
                            for (int vv = v; vv < ve; vv++) {
                                const int ix = ix0 + (vv - v);
                                const Real f = sp[vv];
                                const Real cx = cxhc[ix];
                                const Real t0 = vt[vv * VT] * f;
                                const Real t1 = t0 * cx;
                                const Real t2 = t1 * cx;
                                P0 += t0;
                                P1 += t1;
                                P2 += t2;
                                P3 = fma(t2, cx, P3);
                            }
                            fold(P0, P1, P2, P3, ve);
                            v = ve;
                        }
                    }
                }
            }
            // combine the two halves and write the (group, cell) partial
            using Out = typename PartOut<Real>::T;
            Out *red = reinterpret_cast<Out *>(mred);
            if (vp == 1) {
#pragma unroll
                for (int q = 0; q < NPART; q++) {
                    if constexpr (sizeof(Real) == 8)
                        red[q * SLICE + cl] = S[q].value();
                    else
                        red[q * SLICE + cl] = make_float2(S[q].s, S[q].c);
                }
            }
            __syncthreads();
            if (vp == 0 && valid) {
                // the cell's NPART partials are contiguous (128 bytes)
                Out *pp = COHERENT ? static_cast<Out *>(scratch) + ((size_t)lk * SLICE + cl) * NPART
                                   : static_cast<Out *>(a.part) + ((size_t)vgid * ncell + CELL(GX(li), GY(lj), z)) * NPART;
#pragma unroll
                for (int q = 0; q < NPART; q += 2) {
                    if constexpr (sizeof(Real) == 8) {
                        *reinterpret_cast<double2 *>(pp + q) = make_double2(S[q].value() + red[q * SLICE + cl],
                                                                            S[q + 1].value() + red[(q + 1) * SLICE + cl]);
                    } else {
                        const float2 o0 = red[q * SLICE + cl], o1 = red[(q + 1) * SLICE + cl];
                        const float2 r0 = pair_add(S[q].s, S[q].c, o0.x, o0.y);
                        const float2 r1 = pair_add(S[q + 1].s, S[q + 1].c, o1.x, o1.y);
                        *reinterpret_cast<float4 *>(pp + q) = make_float4(r0.x, r0.y, r1.x, r1.y);
                    }
                }
            }
        }
        // the next slice's halo row overwrites the reduction buffer
        if constexpr (L::red_in_halo) __syncthreads();
    }

    // z outflow of the block for the next stage (own velocities only)
    if (!zlast) {
        for (int cl = 0; cl < SLICE; cl++) {
            const int li = cl % BX, lj = cl / BX;
            if (li >= ex || lj >= ey) continue;
            const int x = GX(li), y = GY(lj);
#pragma unroll
            for (int m = 0; m < TV; m++) {
                if (!ok[m]) continue;
                FZp[((size_t)y * nx + x) * Nv + gv[m]] = slice[SL(li, lj) + t + m * NT];
                if constexpr (ORDER == 2)  // slice ez-2 (the inflow slice k0-1 when ez == 1)
                    FZ2p[((size_t)y * nx + x) * Nv + gv[m]] = slice2[(lj * BX + li) * CS + t + m * NT];
            }
        }
    }
}

// One wavefront stage: CTA (x, y) = (work item x of the stage, velocity group y).
template <typename Real, int TV, int LINE, bool UNIF>
__global__ void __launch_bounds__(NT, 2) sweep_kernel(const SweepArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    sweep_item<Real, TV, LINE, false, UNIF>(a, a.work[blockIdx.x], blockIdx.y, smem, nullptr, nullptr);
}
template <typename Real, int TV, int LINE, bool UNIF, int ORDER, bool DEV>
__global__ void __launch_bounds__(NT, 2) sweep_persistent_kernel(const BatchSweepArgs b)
{
    extern __shared__ __align__(16) unsigned char smem[];
    persistent_loop<Real>(b, [&](const SweepArgs &a, const int4 w, const int vg, void *scratch, Pipe &pipe) {
        sweep_item<Real, TV, LINE, true, UNIF, ORDER, DEV>(a, w, vg, smem, scratch, &pipe);
    });
}

template <typename Real, int TV, int LINE, bool UNIF>
cudaError_t launch_t(const SweepArgs &a, int n_items, int max_vg, cudaStream_t s)
{
    using L = SmemLayout<Real, TV>;
    const size_t bytes = L::total(a.nxo_max, LINE > 0);
    cudaError_t e = ensure_smem(reinterpret_cast<const void *>(sweep_kernel<Real, TV, LINE, UNIF>), bytes);
    if (e != cudaSuccess) return e;
    dim3 grid(n_items, max_vg);
    sweep_kernel<Real, TV, LINE, UNIF><<<grid, NT, bytes, s>>>(a);
    return cudaGetLastError();
}

template <typename Real, int TV>
cudaError_t launch_line(const SweepArgs &a, int n_items, int max_vg, cudaStream_t s)
{
    if constexpr (TV == 1) {
        if (a.line16)
            return a.uniform ? launch_t<Real, TV, 16, true>(a, n_items, max_vg, s)
                             : launch_t<Real, TV, 16, false>(a, n_items, max_vg, s);
    }
    return a.uniform ? launch_t<Real, TV, 0, true>(a, n_items, max_vg, s)
                     : launch_t<Real, TV, 0, false>(a, n_items, max_vg, s);
}

template <typename Real, int TV, int LINE, bool UNIF, int ORDER, bool DEV>
cudaError_t launch_persistent_t(const BatchSweepArgs &b, int nxo_max, int grid, cudaStream_t s)
{
    using L = SmemLayout<Real, TV, ORDER>;
    const size_t bytes = L::total(nxo_max, LINE > 0);
    const void *fn = reinterpret_cast<const void *>(sweep_persistent_kernel<Real, TV, LINE, UNIF, ORDER, DEV>);
    cudaError_t e = ensure_smem(fn, bytes);
    if (e != cudaSuccess) return e;
    sweep_persistent_kernel<Real, TV, LINE, UNIF, ORDER, DEV><<<grid, NT, bytes, s>>>(b);
    return cudaGetLastError();
}

template <typename Real, int TV, int LINE, bool UNIF, int ORDER, bool DEV>
int occupancy_t(size_t smem)
{
    int n = 0;
    const void *fn = reinterpret_cast<const void *>(sweep_persistent_kernel<Real, TV, LINE, UNIF, ORDER, DEV>);
    if (ensure_smem(fn, smem) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sweep_persistent_kernel<Real, TV, LINE, UNIF, ORDER, DEV>,
                                                      NT, smem) != cudaSuccess)
        return 0;
    return n;
}

// Instantiation chosen at run time: one velocity per thread.  The first-order
// FP64 sweep comes here only without the memory for its axis factors
// (k.sep = 0), with the general moment loop alone.
template <template <typename, int, int, bool, int, bool> class F, typename... Args>
auto dispatch(const SweepKind &k, Args &&...args)
{
    if (k.order == 2) {  // one velocity per thread, uniform grids
        if (k.precision == 0)
            return k.line16 ? F<double, 1, 16, true, 2, false>::run(args...)
                            : F<double, 1, 0, true, 2, false>::run(args...);
        return k.line16 ? F<float, 1, 16, true, 2, true>::run(args...) : F<float, 1, 0, true, 2, true>::run(args...);
    }
    if (k.dev) {  // uniform grids
        return k.line16 ? F<float, 1, 16, true, 1, true>::run(args...) : F<float, 1, 0, true, 1, true>::run(args...);
    }
    if (k.precision == 0) {
        return k.uniform ? F<double, 1, 0, true, 1, false>::run(args...)
                         : F<double, 1, 0, false, 1, false>::run(args...);
    }
    if (k.line16)
        return k.uniform ? F<float, 1, 16, true, 1, false>::run(args...)
                         : F<float, 1, 16, false, 1, false>::run(args...);
    return k.uniform ? F<float, 1, 0, true, 1, false>::run(args...) : F<float, 1, 0, false, 1, false>::run(args...);
}

template <typename Real, int TV, int LINE, bool UNIF, int ORDER, bool DEV>
struct PersistentLaunch {
    static cudaError_t run(const BatchSweepArgs &b, int nxo_max, int grid, cudaStream_t s)
    {
        return launch_persistent_t<Real, TV, LINE, UNIF, ORDER, DEV>(b, nxo_max, grid, s);
    }
};

template <typename Real, int TV, int LINE, bool UNIF, int ORDER, bool DEV>
struct Occupancy {
    static int run(size_t smem) { return occupancy_t<Real, TV, LINE, UNIF, ORDER, DEV>(smem); }
};

bool exists(const SweepKind &k)
{
    if (k.tv == 2 && !k.pack) return false;  // two velocities per thread: with packed slots
    if (k.order == 2) return k.tv == 1 && k.uniform;
    return !k.dev || (k.precision != 0 && k.uniform);
}

}  // namespace

int sweep_persistent_occupancy(const SweepKind &k, size_t smem)
{
    if (!exists(k)) return 0;
    if (k.sep) return sweep_d_occupancy(k, smem);
    return k.pack ? sweep2_occupancy(k, smem) : dispatch<Occupancy>(k, smem);
}

cudaError_t launch_sweep_persistent(const SweepKind &k, const BatchSweepArgs &b, int nxo_max, int grid, cudaStream_t s)
{
    if (b.n_items == 0) return cudaSuccess;
    if (!exists(k)) return cudaErrorInvalidValue;
    if (k.sep) return launch_sweep_d(k, b, nxo_max, grid, s);
    return k.pack ? launch_sweep2_persistent(k, b, nxo_max, grid, s) : dispatch<PersistentLaunch>(k, b, nxo_max, grid, s);
}

size_t sweep_smem_bytes(const SweepKind &k, int nxo_max)
{
    if (k.sep) return sweep_d_smem_bytes(k, nxo_max);
    if (k.pack) return sweep2_smem_bytes(k, nxo_max);
    const bool line = k.line16 != 0;
    if (k.order == 2)
        return k.precision == 0 ? SmemLayout<double, 1, 2>::total(nxo_max, line)
                                : SmemLayout<float, 1, 2>::total(nxo_max, line);
    if (k.precision == 0) return SmemLayout<double, 1>::total(nxo_max, false);
    return SmemLayout<float, 1>::total(nxo_max, line);
}

SweepPerSm sweep_per_sm(SweepKind k, int nxo_max)
{
    SweepPerSm n{};
    k.sep = 0;
    n.general = sweep_persistent_occupancy(k, sweep_smem_bytes(k, nxo_max));
    if (k.precision == 0 && k.order == 1) {
        k.sep = 1;
        n.sep = sweep_persistent_occupancy(k, sweep_smem_bytes(k, nxo_max));
    }
    return n;
}

cudaError_t launch_sweep(const SweepKind &k, const SweepArgs &a, int n_items, int max_vg, cudaStream_t s)
{
    if (n_items == 0 || max_vg == 0) return cudaSuccess;
    if (k.pack) return launch_sweep2_staged(k, a, n_items, max_vg, s);
    if (k.precision == 0) return launch_line<double, 1>(a, n_items, max_vg, s);
    if (k.tv == 2) return launch_line<float, 2>(a, n_items, max_vg, s);
    return launch_line<float, 1>(a, n_items, max_vg, s);
}

}  // namespace kgs
