// kgs_internal.h -- device-side data layouts and launch interfaces shared by
// the CUDA translation units of libkgs.  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace kgs {

// Spatial sweep block: BX x BY cells in the XY plane (compile time), a
// run-time number of cells along z.  The XY slice of every in-flight velocity
// stays in shared memory while the block marches along z (Section 3.2's slice
// marching, one slice updated in place).
constexpr int BX = 8;
constexpr int BY = 8;
constexpr int SLICE = BX * BY;
constexpr int NT = 128;          // threads per sweep CTA
constexpr int NCOEF = 16;        // per-cell coefficient record
constexpr int NPART = 16;        // per-cell partial: 13 moment sums + 3 wall fluxes

// Per-cell coefficient record (computed from the lagged FP64 macros each
// iteration, stored in the sweep precision).  U^n below is the lagged velocity
// as rounded to the sweep precision: the centre of c = xi - U^n for the
// moments.  The equilibrium is evaluated from s = |xi|^2 - 2 U^n . xi, which
// is |c|^2 - |U^n|^2; the |U^n|^2 terms are folded into the constants below.
enum {
    C_M2UX = 0, C_M2UY, C_M2UZ,  // -2 U^n (exactly twice the centre, negated)
    C_KAPPA,                // (1/tau) rho (2 pi R T)^{-3/2} exp(-|U^n|^2 / (2RT)); FP32: its base-2 logarithm
    C_NEXP,                 // exponent scale: -1/(2RT) (FP64) or -log2(e)/(2RT) (FP32)
    C_RT1,                  // 1/(R T)
    C_RTAU,                 // 1/tau
    C_FLAGS,                // cell flags (below), their bits stored in the value (flag_value)
    C_QX, C_QY, C_QZ,       // q' = (1 - Pr) q / (5 p R T)
    C_RDX, C_RDY, C_RDZ,    // 1/dx_i, 1/dy_j, 1/dz_k (FP32 second-order sweep, uniform grid:
                            // C_RDX, C_RDY hold the exponent terms of its deviation source)
    C_SHK0,                 // |U^n|^2 / (R T) - 5, so that |c|^2/(RT) - 5 = s/(RT) + C_SHK0
    C_MUQ                   // -U^n . q'
};

// Cell flags.
constexpr int F_SOLID = 1;               // the cell itself is solid
constexpr int F_SOLID_SIDE = 2;          // << s: the neighbour on side s is solid
constexpr int F_WALL_SIDE = 1 << 7;      // << s: face on side s is a diffuse wall

// Partial-sum slots per (velocity group, cell): the 13 sums about U^n
// (S0, S1xyz, S2 xx yy zz xy xz yz, S3xyz) and the incoming flux onto the
// wall ahead of the octant along x, y, z.
enum {
    P_S0 = 0, P_S1X, P_S1Y, P_S1Z, P_S2XX, P_S2YY, P_S2ZZ, P_S2XY, P_S2XZ, P_S2YZ,
    P_S3X, P_S3Y, P_S3Z, P_FX, P_FY, P_FZ
};

// Per-cell sums of one outer iteration as the closure reads them ([NSUM][ncell],
// FP64): the 13 sums about U^n in the P_* order, then the incoming flux onto
// the wall on each domain side s (-x, +x, -y, +y, -z, +z) at slot SUM_F0 + s.
constexpr int SUM_F0 = 13;
constexpr int NSUM = 19;
// Ordered accumulators of the persistent sweep: [nacc][ncell][acc_slots] (FP64,
// or float-float pairs (hi, lo) for the FP32 path).  ACC_COMPACT slots: the
// 13 sums, then one incoming flux per axis -- the flux onto the only wall a
// cell has along that axis -- the layout of an item's partials, so that an
// item adds its record element-wise.  ACC_SPLIT slots: the 13 sums, then one
// flux per side (slot SUM_F0 + side), for problems where some cell has walls
// on both sides along an axis.
constexpr int ACC_COMPACT = 16;
constexpr int ACC_SPLIT = 20;
constexpr int NACC_MAX = 8;  // accumulators per instance, at most

// Reference Maxwellian of the FP32 sweep, which carries g = f - M_ref rather
// than f: the moments of the FP32 table values of M_ref over the swept
// velocities, raw[a][b][c] = sum w M_ref xi_x^a xi_y^b xi_z^c (a + b + c <= 3,
// index ref_index), and their incoming flux onto each domain side.  All zero
// for the FP64 path, which carries f itself.
constexpr int NREF = 20;
__host__ __device__ constexpr int ref_index(int a, int b, int c)
{
    // a + b + c = n occupies [n (n+1) (n+2) / 6, ...), ordered by (b + c, c)
    return (a + b + c) * (a + b + c + 1) * (a + b + c + 2) / 6 + (b + c) * (b + c + 1) / 2 + c;
}
struct RefMoments {
    double raw[NREF];
    double flux[6];
};

// Wall-Maxwellian table rows: 0..5 domain side, 6 solid surface, 7 free stream.
constexpr int MT_SOLID = 6;
constexpr int MT_INFLOW = 7;
constexpr int MT_ROWS = 8;

struct SweepArgs {
    int nx, ny, nz, bz;           // grid, block extent along z
    int nbx, nby, nbz;            // blocks per axis
    const int4 *work;             // per CTA row: octant, reflected block coords
    const int *oct_vstart;        // [8] first velocity slot of each octant
    const int *oct_vcount;        // [8] velocities per octant
    const int *oct_vgbase;        // [8] first global velocity-group index
    int Nv;                       // all velocity slots
    int vg_size;                  // velocities per CTA
    const void *vel;              // Real[Nv][4]: xi_x, xi_y, xi_z, w (octant-sorted)
    const void *velm;             // Real[Nv][8]: w_x, w_y w_z, the low parts of xi_x, xi_y, xi_z
                                  // (xi = hi + lo with hi = the value in vel), M_ref (FP32
                                  // path; 0 for FP64), the rounding error of M_ref and
                                  // |xi|^2 of the rounded node (FP32 path)
    int pack;                     // packed velocity slots (HostTables::pack, FP32 with two velocities per thread)
    int oct_line0[8];             // packed: first row of each octant in lines
    const float *lines;           // packed: [lines][8] xi_y, xi_z, w_y w_z, low parts of xi_y, xi_z
    const float *xnodes;          // packed: [8][xn_stride][4] xi_x, its low part, w_x
    int xn_stride;
    int oct_nx[8];                // x nodes in each octant (length of its velocity x-lines)
    int oct_ny[8];                // y nodes in each octant (x-lines per velocity plane)
    const void *ax_tab;           // separated FP64 sweep: double4[ncell][ax_n] axis factors (kgs_sweep_d.cu)
    int ax_n, ax_nx, ax_ny;       // nodes of the three axes, of x and of y, in HostTables::ax_nodes order
    int ax_neg[3];                // negative nodes of each axis (they come first)
    const double *centre;         // separated FP64 sweep: [nz][nby][nbx][4] the velocity about which the sums of
                                  // the cells of one block's slice are taken and, if not 0 in the fourth place,
                                  // that each cell's are about its own U^n instead (slice_centre)
    int nxo_max;                  // max over octants of oct_nx
    int any_solid;                // the problem has solid cells
    const uint8_t *blk_plain;     // [nbz][nby][nbx]: 1 = no solid cell and no solid neighbour in the block (or NULL)
    const void *coef;             // Real[ncell][NCOEF]
    const double *rho_w;          // [6][ncell]
    const float *rho_w32;         // the same in FP32 (persistent packed FP32 sweep)
    const void *mtab;             // Real[MT_ROWS][Nv]: unit wall Maxwellians, free stream
    int side_inflow[6];           // domain side s is a free-stream boundary
    void *FX, *FY, *FZ;           // face planes: [nz*ny][Nv], [nz*nx][Nv], [ny*nx][Nv]
    int order;                    // upwind order of the sweep (1: Eq. (7), 2: three-point differences)
    void *FX2, *FY2, *FZ2;        // order 2: the planes one cell further upwind (same shapes)
    void *part;                   // staged sweep: [n_vg][ncell][NPART], double (FP64 path) or
                                  // float2 (s, c) with value s - c (FP32 path, Kahan pair)
    void *acc;                    // persistent sweep: [nacc][ncell][acc_slots] ordered accumulators
    int nacc;                     // accumulators: velocity group g (of all groups) adds into g % nacc
    int acc_slots;                // ACC_COMPACT or ACC_SPLIT
    int *tok;                     // persistent sweep: [nacc][nbz][nby][nbx] chain tokens
    unsigned long long ncell;
    int line16;                   // every octant has x-lines of 16 nodes (specialised moment loop)
    int uniform;                  // equal cell widths along each axis: a_d is per velocity
    double rd0[3];                // 1/dx, 1/dy, 1/dz of a uniform grid
};

// Persistent sweep over the work items of many instances (one launch per
// outer iteration): item = (instance, octant << 24 | velocity group of the
// octant, reflected block coordinates bx | by << 10 | bz << 20, global
// velocity-group index within the instance), list ordered by stage.
struct BatchSweepArgs {
    const SweepArgs *inst;        // [n_inst] per-instance arguments (device)
    const int4 *items;
    int n_items;
    int *counter;                 // claim counter, zero at launch
    int *flags;                   // progress of each item, zero at launch
    const int *flag_off;          // [n_inst] first flag of each instance
    const int *pos;               // [n_items] place of each item in its accumulator chain
    void *scratch;                // [grid][bz * SLICE][NPART] per-CTA moment partials
    unsigned long long scratch_stride;  // bytes of one CTA's scratch, sweep_scratch_bytes(bz)
    int *error;                   // set to 1 when a bounded wait gives up
    long long spin_limit;         // polls before a wait gives up
    int skip_publish;             // fault injection: this item never sets its flag (-1: none)
    int announce_every;           // slices between two announcements of an item's progress (announce_every())
};
// A block that announces its progress lets its x and y neighbours overlap
// with it, at the price of a release (which waits for the block's stores) per
// announcement.  FP64 slices take 20 us or more and announce each.  FP32 slices
// take 6 to 12 us: measured times per iteration with an announcement every 1 /
// 2 / 8 slices or only at the end are 392 / 412 / 545 / 734 us for 64 items
// (16^3 cells x 16^3 velocities), 3.66 / 3.66 / 3.74 / 5.3 ms for 2520 items
// (45 x 38 x 41 x 22 x 19 x 24) and 19.44 / 19.33 / 19.26 / 19.3 ms for 16384
// (64^3 x 32^3), on 304 resident blocks.
inline int announce_every(int precision, int n_items, int grid)
{
    if (precision == 0 || n_items <= grid) return 1;
    return n_items <= 16 * grid ? 2 : 8;
}
// Bytes of one CTA's scratch partials for blocks bz cells deep (both precisions
// store 8 bytes per slot).
inline size_t sweep_scratch_bytes(int bz) { return (size_t)bz * SLICE * NPART * 8; }

// Cell flags travel in the coefficient array as the bit pattern of a Real
// (no conversion instruction on either side).
__host__ __device__ inline float flag_value_f(int f)
{
    union {
        int i;
        float v;
    } u;
    u.i = f;
    return u.v;
}
__host__ __device__ inline double flag_value_d(int f)
{
    union {
        long long i;
        double v;
    } u;
    u.i = f;
    return u.v;
}
template <typename Real>
__host__ __device__ inline Real flag_value(int f);
template <>
__host__ __device__ inline float flag_value<float>(int f)
{
    return flag_value_f(f);
}
template <>
__host__ __device__ inline double flag_value<double>(int f)
{
    return flag_value_d(f);
}
__device__ __forceinline__ int flag_bits(float v) { return __float_as_int(v); }
__device__ __forceinline__ int flag_bits(double v) { return (int)__double_as_longlong(v); }

// Which sweep kernel serves a problem.
struct SweepKind {
    int precision = 0;            // 0 FP64, 1 FP32
    int tv = 1;                   // velocities per thread (FP64, order 2: 1)
    int line16 = 0;               // SweepArgs::line16
    int uniform = 0;              // SweepArgs::uniform
    int order = 1;                // upwind order; order 2 exists for tv = 1 on uniform grids only
    int dev = 0;                  // first-order FP32 sweep with the deviation-form source (uniform grids)
    int pack = 0;                 // SweepArgs::pack: the packed FP32 kernel (kgs_sweep_f2.cu)
    int lines_max = 1;            // x-lines that a velocity group can touch, at most
    int sep = 0;                  // first-order FP64 sweep with separated equilibria (kgs_sweep_d.cu)
};
// Persistent sweep.  Combinations that do not exist: 0 CTAs per SM /
// cudaErrorInvalidValue.
cudaError_t launch_sweep_persistent(const SweepKind &k, const BatchSweepArgs &b, int nxo_max, int grid,
                                    cudaStream_t s);
// Resident CTAs per SM of the persistent kernel (also sets its shared-memory limit).
int sweep_persistent_occupancy(const SweepKind &k, size_t smem);
size_t sweep_smem_bytes(const SweepKind &k, int nxo_max);
// The two of them for the kernel that needs no axis factors and for the
// separated one (0 where it does not apply or its tables do not fit).
struct SweepPerSm {
    int general, sep;
};
SweepPerSm sweep_per_sm(SweepKind k, int nxo_max);
// Sweep launch (one wavefront stage, order 1, no deviation-form source).
cudaError_t launch_sweep(const SweepKind &k, const SweepArgs &a, int n_items, int max_vg, cudaStream_t s);

// The separated FP64 kernel (k.sep), reached through the functions above, and
// the axis factors that it reads, from the FP64 cell coefficients.
size_t sweep_d_smem_bytes(const SweepKind &k, int nxo_max);
int sweep_d_occupancy(const SweepKind &k, size_t smem);
cudaError_t launch_sweep_d(const SweepKind &k, const BatchSweepArgs &b, int nxo_max, int grid, cudaStream_t s);
cudaError_t launch_axis_tables(const void *coef, const double *nodes, unsigned long long ncell, int nvx, int nvy,
                               int na, void *tab, cudaStream_t s);
cudaError_t launch_slice_centres(const void *coef, int nx, int ny, int nz, double *centre, cudaStream_t s);
// Entry of SweepArgs::centre for cell (i, j, k) of an nx x ny x nz grid.
__host__ __device__ inline size_t slice_centre(int i, int j, int k, int nx, int ny)
{
    const int nbx = (nx + BX - 1) / BX, nby = (ny + BY - 1) / BY;
    return (((size_t)k * nby + j / BY) * nbx + i / BX) * 4;
}

// The packed FP32 kernels (k.pack), reached through the functions above.
size_t sweep2_smem_bytes(const SweepKind &k, int nxo_max);
int sweep2_occupancy(const SweepKind &k, size_t smem);
cudaError_t launch_sweep2_persistent(const SweepKind &k, const BatchSweepArgs &b, int nxo_max, int grid,
                                     cudaStream_t s);
cudaError_t launch_sweep2_staged(const SweepKind &k, const SweepArgs &a, int n_items, int max_vg, cudaStream_t s);

// Per-cell sums of the staged sweep's per-group partials (fixed group order).
struct PartSumArgs {
    unsigned long long ncell;
    int n_vg;
    const int *vg_oct;            // [n_vg] octant of each velocity group
    const void *part;             // [n_vg][ncell][NPART], see SweepArgs::part
    int precision;
    const uint8_t *solid;         // [ncell] or NULL
    double *sums;                 // [NSUM][ncell]
    const void *coef;             // sweep-precision coefficients (U centre)
    const int8_t *wall_kind;      // [6][ncell]
    RefMoments ref;               // moments of the reference Maxwellian, added to every cell
};

// What the closure and the residual kernel of an iteration pass on; all zero
// before the first iteration.
struct CloseState {
    unsigned closed, checked;     // blocks of either kernel that have finished (zero between launches)
    double mass;                  // total mass, of a closure of many blocks
};
struct ClosureArgs {
    int nx, ny, nz;
    unsigned long long ncell;
    const double *sums;           // [NSUM][ncell]
    const void *coef;             // sweep-precision coefficients (U centre)
    int precision;
    int q_lagged;                 // 1: q = S3 / 2 about the lagged U^n (no shift)
    double *mac_new;              // [8][ncell] step n+1 (before rescale)
    double *rho_w_new;            // [6][ncell]
    const int8_t *wall_kind;      // [6][ncell]: -1 not a wall, 0..6 wall kind
    const double *wall_norm;      // [7][6] rho_w = F * wall_norm[kind][side]
    const double *dx, *dy, *dz;
    const uint8_t *solid;         // [ncell] or NULL
    double *blk_mass;             // [close_blocks(ncell)]
    int rescale;                  // the mass is wanted
    CloseState *state;
};

// dev_src (FP32 only): the C_RDX / C_RDY slots carry the exponent terms of
// the second-order sweep's deviation source instead of 1/dx, 1/dy.  rho_w32
// (may be NULL) receives rho_w [6][ncell] rounded to FP32.
cudaError_t launch_coef(int precision, const double *mac, const uint8_t *solid, const uint8_t *cell_flags_side,
                        const double *rdx, const double *rdy, const double *rdz, int nx, int ny, int nz,
                        double mu_ref, double omega, double Pr, void *coef, cudaStream_t s, int dev_src = 0,
                        const double *rho_w = nullptr, float *rho_w32 = nullptr);
// Cells per block of the closure kernel; blk_mass holds close_blocks(ncell)
// values.
constexpr int CLOSE_CELLS = 32;
inline size_t close_blocks(size_t ncell) { return (ncell + CLOSE_CELLS - 1) / CLOSE_CELLS; }
cudaError_t launch_part_sums(const PartSumArgs &a, cudaStream_t s);
// Per-cell sums of the persistent sweep's ordered accumulators (fixed order).
struct AccSumArgs {
    int precision;
    const void *acc;
    int nacc;
    int acc_slots;
    const double *centre;         // FP64: about what the accumulated sums are (SweepArgs::centre); NULL: about U^n
    int nx, ny;
    unsigned long long ncell;
    const uint8_t *solid;         // [ncell] or NULL
    double *sums;                 // [NSUM][ncell]
    const void *coef;             // sweep-precision coefficients (U centre)
    const int8_t *wall_kind;      // [6][ncell]
    RefMoments ref;
};
cudaError_t launch_acc_sums(const AccSumArgs &a, cudaStream_t s);
cudaError_t launch_closure(const ClosureArgs &a, cudaStream_t s);
// launch_acc_sums and launch_closure in one, the sums kept in registers;
// blk_mass receives acc_close_blocks(ncell) values.
cudaError_t launch_acc_close(const AccSumArgs &a, const ClosureArgs &k, cudaStream_t s);
unsigned long long acc_close_blocks(unsigned long long ncell);
// Rescale, divergence check and residual after a closure.
struct ResidualArgs {
    double *mac_new, *rho_w_new;  // step n+1, rescaled in place
    const double *mac;            // step n
    const uint8_t *solid;         // [ncell] or NULL
    unsigned long long ncell;
    double M0;
    int rescale;                  // 1: scale the total mass to M0
    double *blk_res;              // [blocks of 256 cells][10]
    int *blk_bad;                 // [blocks of 256 cells]
    const double *blk_mass;       // [n_mass] of the closure, if rescale
    int n_mass;
    CloseState *state;
    double *out;                  // residual, divergence flag
};
cudaError_t launch_residual(const ResidualArgs &a, cudaStream_t s);
cudaError_t launch_wall_flux_init(const double *mac, const int8_t *wall_kind, const double *wall_norm,
                                  const double *axis64, int nvx, int nvy, int nvz, unsigned long long ncell, double R,
                                  double Pr,
                                  double *rho_w, cudaStream_t s);

}  // namespace kgs
