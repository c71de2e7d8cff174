// Private declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <cmath>

#include <nvtx3/nvToolsExt.h>

#include "lb.h"

namespace lbm {

// NVTX range over the host side of an entry point (named in profiler timelines; a few
// nanoseconds when no tool is attached).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// An error that a call returns is reported: it does not stay behind as the runtime's last error, which
// the next launch of this host thread, of any context, would take for its own.
inline lb_status reported(lb_status s) {
    if (s == LB_ECUDA || s == LB_ENOMEM) (void)cudaGetLastError();
    return s;
}

// Error bits written by kernels into the context's device flag word.
enum : int { ERR_DOMAIN = 1, ERR_TIMEOUT = 2 };

// Order of the population planes in a stored state buffer: grouped by the row each
// population is pulled from in a step (f_a(x, y) = g_a(x - e_a)): the planes of 2, 5, 6
// (pulled from row y - 1), then 0, 1, 3 (row y), then 4, 7, 8 (row y + 1). Population a of
// the state lives in plane plane_of(a); host arrays keep the natural order 0..8.
__host__ __device__ constexpr int plane_of(int a) {
    return a == 2 ? 0 : a == 5 ? 1 : a == 6 ? 2 : a == 0 ? 3 : a == 1 ? 4 : a == 3 ? 5
         : a == 4 ? 6 : a;
}

// Elements in front of column 0 of every stored row (the last two hold periodic images or
// edge copies). FP32 uses 8, so that column 0 sits 32 bytes into the row and each warp's
// 64-column store covers whole 32-byte sectors; the TMA box (columns x0 - 4 ..) then starts
// at element x0 + 4, still 16-byte aligned. FP64 rows are sector-aligned with 4 already,
// and BF16 keeps 4 because its box start must stay a multiple of 8 elements.
constexpr int ghost_of_prec(int prec) { return prec == LB_FP32 ? 8 : 4; }

// Per-lattice constants of the update, in double; kernels convert them to their type.
struct Consts {
    int eos_kind;
    // Carnahan-Starling: p = rho RT (1 + eta + eta^2 - eta^3)/(1 - eta)^3 - a rho^2, eta = b4 rho
    double a, b4, RT;
    // exponential potential psi0 exp(-rho0/rho)
    double psi0, rho0;
    // Eq. 23 branches; p_rho1 = rho1 th_v, p_rho2 = p_rho1 + (rho2 - rho1) th_m
    double th_v, th_m, th_l, rho1, rho2, p_rho1, p_rho2;
    // psi^2 = (p - rho/3) * two_over_G for the EOS-based potentials
    double two_over_G;
    double G;       // interaction strength of Eq. 7
    double kG2;     // kappa G / 2 of Eq. 19
    double sig_coef;  // 12 sigma G^2 / (tau_e - 1/2): Eq. 8 with |F|^2/psi^2 = G^2 |sum w psi e|^2
    double s_e, s_z, s_q, s_v;  // non-conserved relaxation rates (s_rho, s_j drop out, see kernels)
    int stall_row;  // test hook: the kernels wait for this row in vain (INT_MIN = off)
    double shift_rho;  // rho_s of the LB_BF16 storage shift f_a - w_a rho_s (0 otherwise)
    int stochastic;    // LB_BF16: 1 = stochastic rounding of the stored values (0 = nearest)
    unsigned step_key; // the step a launch takes (the stochastic-rounding counter)
    // nu(rho) of the open-boundary kernels: s_v_vapour where rho < rho_sw (-inf: off)
    double rho_sw, s_v_vapour;
};

// Geometry of one lattice's device population buffer.
struct Geom {
    int nx, ny;
    int pitch;          // elements per stored row (>= nx + 2 * ghost, multiple of 32)
    long long plane;    // elements per population plane = ny * pitch
    int walls;          // boundary kind (lb_bc): 0 periodic, 1 walls in y, 2 open (see lb.h)
};

// One work item of the batched step: a strip of one lattice.
struct BatchItem {
    int lat;            // lattice index
    int x0, w;          // first column (a multiple of 4) and width (<= the kernel's TX)
    int yb, n, dir;     // first row, row count, march direction (+1 / -1)
};

// Lattices that the direct batched step takes in one launch (a kernel parameter: what a CTA needs
// to start its loads comes from the constant bank).
constexpr int GROUP_LATTICES = 64;
struct BatchGroup {
    struct Lattice {
        void *g[2];         // the lattice's two population buffers
        int nx, ny, pitch;
        unsigned plane;
        int tiles_x, lat;
    } l[GROUP_LATTICES];
};

// One CTA's share of a batched measurement: rows row0 .. row0 + rows - 1 of a lattice.
struct MeasureChunk {
    int lat, row0, rows;
};

struct StepLaunch {
    int variant;        // compiled (strip width, ring depth) choice, see step_variant_tx
    int tx;             // lattice columns per CTA (two per thread)
    int rows;           // rows each CTA marches over
    int ctas_per_sm;    // resident CTAs per SM reported by the occupancy calculator (ring variants; the
                        // others' rows do not depend on it, see tile_occupancy)
};

// ---- kernels (lb_kernels.cu) -------------------------------------------------------
int step_variant_count();
int direct_variant();                   // the variant of the direct kernels (lb_tile.cuh)
int staged_variant();                   // their TMA-staged tiles (LB_FP32 and LB_BF16)
bool direct_fits(const Geom &g);        // the direct kernels' grid holds the lattice
int default_variant(int prec, const Geom &g);   // what a context starts with
// tiles of the direct and of the staged FP32 and BF16 kernels
constexpr int DIRECT_COLS = 64, DIRECT_ROWS = 4, STAGED_ROWS = 4;
// the staged tile's TMA box: columns x0 - 4 .. x0 + 67 (a 16-byte aligned start in both types), the
// rows of the tile and one on either side, three planes
constexpr int TILE_BOX_LEFT = 4, TILE_BOX_W = DIRECT_COLS + 8, TILE_BOX_ROWS = STAGED_ROWS + 2;
// whether the staged kernel brings the tile of rows y0 .. y0 + r - 1 into shared memory: not where rows
// wrap, nor where the row above the tile is the last below a wall (it bounces populations of its own
// row, which its plane group's box does not reach)
__host__ __device__ constexpr bool tile_staged(int bc, int y0, int r, int ny) {
    return bc == 0 ? y0 >= 2 && y0 + r + 2 <= ny : !(bc == 1 && y0 + r == ny - 1);
}
bool staged_loads_row(const Geom &g, int row);      // some staged tile's boxes hold this lattice row
bool resident_waits_for_row(const Geom &g, int row);   // some tile has it beside it (lb_resident.cu)
int step_variant_tx(int variant);
int step_variant_planes(int variant);   // population planes per TMA box (9 or 3)
int default_ring_variant();
StepLaunch make_step_launch(int prec, int eos_kind, const Geom &g, int num_sms, int variant,
                            int rows_override);
cudaError_t configure_step(int prec, const Consts &c, const Geom &g, const StepLaunch &l);
// tensor_map_in: a CUtensorMap describing the input buffer (3-D: x, y, population plane).
// Step units, one per storage type and ring kind K (lb_step_<type>.cu: K = 0, whole-row
// ring; lb_step_<type>_stage.cu: K = 1, stage ring); configure: set the kernel attributes
// only. A variant of the other kind returns cudaErrorInvalidValue (occupancy 0).
#define LB_DECLARE_STEP_UNIT(NAME, K)                                                         \
    cudaError_t step_##NAME##_k##K(const Consts &c, const Geom &g, const StepLaunch &l,      \
                                   int order, const void *tensor_map_in, void *gout, int *err, \
                                   cudaStream_t st, bool configure);                         \
    int occupancy_##NAME##_k##K(int variant, int eos_kind, int bc);
LB_DECLARE_STEP_UNIT(f32, 0)
LB_DECLARE_STEP_UNIT(f32, 1)
LB_DECLARE_STEP_UNIT(f64, 0)
LB_DECLARE_STEP_UNIT(f64, 1)
LB_DECLARE_STEP_UNIT(bf16, 0)
LB_DECLARE_STEP_UNIT(bf16, 1)
#undef LB_DECLARE_STEP_UNIT
int step_variant_kind(int variant);   // 0: whole-row ring, 1: stage ring
// batched-step units (lb_batch_kernels.cu: K = 0, lb_batch_stage.cu: K = 1)
#define LB_DECLARE_BATCH_UNIT(NAME, K)                                                        \
    cudaError_t batch_##NAME##_k##K(int variant, int eos, bool configure, int *occ, int grid, \
                                    const void *maps, const void *lats, const BatchItem *items, \
                                    int n_items, int phase, int *errs, cudaStream_t st);
LB_DECLARE_BATCH_UNIT(f32, 0)
LB_DECLARE_BATCH_UNIT(f32, 1)
LB_DECLARE_BATCH_UNIT(f64, 0)
LB_DECLARE_BATCH_UNIT(f64, 1)
#undef LB_DECLARE_BATCH_UNIT

// direct step units (lb_split_f64.cu, lb_batch_tile.cu; lb_tile_f32.cu and lb_tile_bf16.cu below);
// StepBuffers::psi: ny * pitch elements
struct StepBuffers;
cudaError_t split_f64(const Consts &c, const Geom &g, const StepBuffers &b, int *err, cudaStream_t st);

// n lattices of a group, at most max_tiles tiles each
cudaError_t batch_tile_f32(int eos, const BatchGroup &group, int n, int max_tiles, const void *maps,
                           const void *lats, int phase, int *errs, cudaStream_t st);

// n_steps steps of a mid-size lattice in one launch (lb_resident.cu), with `words` of resident_bytes
// bytes, zero before the first launch (resident_bytes 0: the lattice does not fit)
size_t resident_bytes(int prec, const Consts &c, const Geom &g, int num_sms);
cudaError_t launch_resident_steps(const Consts &c, const Geom &g, int num_sms, const void *gin, void *gout,
                                  int n_steps, void *words, int *err, cudaStream_t st);

// n_steps steps of a small lattice in one launch (lb_cluster.cu); cluster_fits: whether it can
bool cluster_fits(int prec, const Consts &c, const Geom &g);
cudaError_t launch_cluster_steps(const Consts &c, const Geom &g, const void *gin, void *gout,
                                 int n_steps, int *err, cudaStream_t st);

// What a step reads and writes: the input buffer and its tensor map (none for the direct FP64
// kernels), the output buffer, and psi scratch (direct FP64 kernels only). occ (variants 7 and 8): not
// launched, the smallest of *occ and the kernels' resident CTAs per SM goes there.
struct StepBuffers {
    const void *gin;
    const void *tensor_map_in;
    void *gout;
    void *psi;
    int *occ = nullptr;
};
int tile_occupancy(int prec, const Consts &c, const Geom &g, int variant);   // of variants 7 and 8
cudaError_t tile_f32(const Consts &c, const Geom &g, int variant, int order,
                     const StepBuffers &b, int *err, cudaStream_t st);
cudaError_t tile_bf16(const Consts &c, const Geom &g, int variant, int order,
                      const StepBuffers &b, int *err, cudaStream_t st);
// order 0 / 1: visit the row blocks (and the rows inside them) forward / in reverse
cudaError_t launch_step(int prec, const Consts &c, const Geom &g, const StepLaunch &l, int order,
                        const StepBuffers &b, int *err, cudaStream_t stream);
// packed: f in the host layout [a][y][x] (no pitch, no ghosts) instead of the padded one
cudaError_t launch_unstream(int prec, const Geom &g, const void *f, void *gbuf, bool packed,
                            cudaStream_t stream);
cudaError_t launch_stream(int prec, const Geom &g, const void *gbuf, void *f, bool packed,
                          cudaStream_t stream);
cudaError_t launch_init_feq(int prec, const Consts &c, const Geom &g, const double *rho,
                            const double *ux, const double *uy, void *f, int *err,
                            cudaStream_t stream);
// psi: nx*ny elements of the storage type
cudaError_t launch_psi_field(int prec, const Consts &c, const Geom &g, const void *gbuf,
                             void *psi, int *err, cudaStream_t stream);
cudaError_t launch_macro_fields(int prec, const Consts &c, const Geom &g, const void *gbuf,
                                const void *psi, double *rho, double *ux, double *uy,
                                cudaStream_t stream);
// Words of a context that its kernels write into host memory: after a wait for the
// stream the host reads them, without a copy. Error bits are written only when there is an error.
struct HostWords {
    int err;
    double out8[8];
};

// Deterministic FP64 reductions; partials must hold 8 * reduce_blocks(n) doubles, ticket is a device
// word that is zero between launches. Results in out (host or device memory): mass, momentum, max
// |v|^2 (4 doubles), and the Laplace sums of a droplet (8 doubles, layout of k_droplet_sums).
int reduce_blocks(long long n_sites);
cudaError_t launch_macro_reduce(int prec, const Consts &c, const Geom &g, const void *gbuf,
                                const void *psi, double *partials, unsigned *ticket,
                                double *out, cudaStream_t stream);
cudaError_t launch_droplet_sums(int prec, const Consts &c, const Geom &g, const void *gbuf,
                                double r_in, double r_out, double *partials, unsigned *ticket,
                                double *out, cudaStream_t stream);
// interface height of every column into h (nx doubles); first: nx ints of scratch
cudaError_t launch_interface_height(int prec, const Consts &c, const Geom &g, const void *gbuf,
                                    double rho_mid, int *first, double *h, cudaStream_t stream);

// Squared distances from the lattice centre ((nx-1)/2, (ny-1)/2) are quarters of integers
// D = (2x - nx + 1)^2 + (2y - ny + 1)^2, so r < r_in is D < quarters_below(r_in) and r > r_out is
// D >= quarters_above(r_out) exactly as with r = sqrt(D / 4), without a root per site.
__host__ __device__ inline long long quarters_below(double r) {   // smallest D with sqrt(D / 4) >= r
    if (!(r > 0)) return 0;
    if (r > 1e9) return 0x7fffffffffffffffll;
    long long d = (long long)(4.0 * r * r);
    while (d > 0 && sqrt(0.25 * (double)(d - 1)) >= r) --d;
    while (sqrt(0.25 * (double)d) < r) ++d;
    return d;
}
__host__ __device__ inline long long quarters_above(double r) {   // smallest D with sqrt(D / 4) > r
    if (r < 0) return 0;
    if (!(r <= 1e9)) return 0x7fffffffffffffffll;
    long long d = (long long)(4.0 * r * r);
    while (d > 0 && sqrt(0.25 * (double)(d - 1)) > r) --d;
    while (!(sqrt(0.25 * (double)d) > r)) ++d;
    return d;
}

// Laplace-law results from the 8 sums of a droplet measurement (the layout of
// lb_batch_measure / lb_measure_droplet's out): theta, rho_in, rho_out, R (from the mass),
// p_in, p_out, mass, failed
inline void droplet_results(const double m[8], double n_sites, bool failed, double o[8]) {
    const double rho_in = m[2] > 0 ? m[1] / m[2] : NAN;
    const double rho_out = m[4] > 0 ? m[3] / m[4] : NAN;
    const double p_in = m[2] > 0 ? m[5] / m[2] : NAN;
    const double p_out = m[4] > 0 ? m[6] / m[4] : NAN;
    const double R = std::sqrt((m[0] - rho_out * n_sites) /
                               (3.14159265358979323846 * (rho_in - rho_out)));
    o[0] = (p_in - p_out) * R;
    o[1] = rho_in;
    o[2] = rho_out;
    o[3] = R;
    o[4] = p_in;
    o[5] = p_out;
    o[6] = m[0];
    o[7] = (failed || m[7] > 0 || !std::isfinite(o[0])) ? 1.0 : 0.0;
}

// ---- batched step (lb_kernels.cu) --------------------------------------------------------
// maps: 2 CUtensorMap per lattice (buffer 0, buffer 1); lats: BatchLattice<T> table
cudaError_t configure_batch(int prec, int eos_kind, int variant, int *ctas_per_sm);
cudaError_t launch_batch_step(int prec, int eos_kind, int variant, int grid, const void *maps,
                              const void *lats, const BatchItem *items, int n_items, int phase,
                              int *errs, cudaStream_t stream);
// per lattice: out[8*i ..] = mass, sum rho (r < R/2), count, sum rho (outside), count,
// sum p (inside), sum p (outside), non-finite count; FP64, fixed order. Lattice i is measured
// by chunks first[i] .. first[i+1] - 1; partials: 8 * n_chunks doubles
cudaError_t launch_batch_measure(int prec, int eos_kind, const void *lats, int n_lat,
                                 const MeasureChunk *chunks, const int *first, int n_chunks,
                                 int phase, const double *radius, double *partials, double *out,
                                 cudaStream_t stream);

// ---- read-only view of a context for entry points outside lb_api.cu (lb_noalloc.cu) ---
struct CtxView {
    const void *g;        // device buffer holding the current state
    Geom geom;
    Consts consts;
    int prec;
    cudaStream_t stream;
    lb_status sticky;
};
lb_status ctx_view(const lb_ctx *c, CtxView *v);
// record a message; with poison = true also make `s` the context's sticky status
lb_status ctx_fail(lb_ctx *c, lb_status s, const char *msg, bool poison);
// wait for the context's stream and fold the device error bits that its kernels set
// (ERR_TIMEOUT, ERR_DOMAIN) into its sticky status, exactly as every synchronising entry
// point of lb_api.cu does; allocates nothing
lb_status ctx_sync_check(lb_ctx *c);

// ---- host thermodynamics (lb_thermo.cpp) ---------------------------------------------
double p_eos_host(const lb_eos &e, double G, double rho);

}  // namespace lbm
