// C ABI of the library (declared in include/lb.h): context management, argument
// validation, device buffers, TMA descriptors and the host side of every call.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>

#include "lb_internal.h"

using lbm::Consts;
using lbm::Geom;

struct lb_ctx {
    Geom geom{};
    Consts consts{};
    int prec = LB_FP64;
    size_t elem = 8;
    cudaStream_t stream = nullptr;
    void *f[2] = {nullptr, nullptr};
    alignas(64) CUtensorMap tmap[2];  // TMA descriptors of f[0] and f[1]
    bool own_f = false;
    int cur = 0;                 // buffer holding the current state g (f = pull of g)
    int num_sms = 0;
    lbm::HostWords *words = nullptr;   // host memory: error bits and reduction results (make_words)
    bool words_locked = false;         // page-locked by the runtime
    int *d_err = nullptr;        // = &words->err, as the kernels address it
    double *d_out8 = nullptr;    // = words->out8, as the kernels address it
    unsigned *d_ticket = nullptr;      // of the reductions (behind d_partials)
    double *d_field = nullptr;   // diagnostics: two nx*ny double fields
    double *d_partials = nullptr;  // 8 doubles per reduction block
    int *d_first = nullptr;        // interface height: nx ints
    double *d_host_in = nullptr; // 3*nx*ny staging for lb_set_rho_u
    void *d_psi = nullptr;       // FP64 direct kernels: psi of the step, ny * pitch elements
    lbm::StepLaunch launch{};
    int asked_variant = 0, asked_rows = 0;   // what apply_launch was last asked for
    bool asked_many = false;
    int many = 0;                // several steps at once: 1 the cluster kernel, 2 the resident one
    void *d_words = nullptr;     // exchange words of the resident kernel
    long long steps = 0;
    long long launches = 0;      // kernel launches that lb_step has queued
    lb_status sticky = LB_OK;
    std::string msg;
};

namespace {

const char *kNoCtx = "no context";
// Most steps of one launch of the cluster or the resident kernel, and the fewest (lb_ctx::many). Such
// a launch loads the lattice, and the resident kernel sets up its exchange, for the time of several
// single steps: together / singly, us, cluster kernel: 64^2 2 steps 11.6 / 5.7, 6 15.4 / 13.7, 7 15.5 /
// 15.8, 24 30 / 51; resident kernel: 501 x 383 2 steps 21.9 / 10.1, 8 40.3 / 36.9, 10 46.4 / 45.9, 12 52.5
// / 55.1, 24 89 / 108; 600 x 225 splash 10 43.8 / 43.3, 24 87 / 102. The lines lie where the first
// lattice gains; others gain later (128^2 from 20 steps on, 512^2 from 35).
constexpr int kManySteps = 1024;
constexpr int kManyLeast[3] = {0, 7, 10};

lb_status fail(lb_ctx *c, lb_status s, const std::string &m) {
    if (c) c->msg = m;
    return lbm::reported(s);
}

lb_status poison(lb_ctx *c, lb_status s, const std::string &m) {
    c->sticky = s;
    c->msg = m;
    return s;
}

lb_status cuda_fail(lb_ctx *c, cudaError_t e, const char *where) {
    std::string m = std::string(where) + ": " + cudaGetErrorString(e);
    return fail(c, LB_ECUDA, m);
}

#define LB_CUDA(ctx, call)                                        \
    do {                                                          \
        cudaError_t e__ = (call);                                 \
        if (e__ != cudaSuccess) return cuda_fail(ctx, e__, #call); \
    } while (0)

size_t elem_size(int prec) { return prec == LB_FP32 ? 4 : (prec == LB_BF16 ? 2 : 8); }

bool rate_ok(double s) { return std::isfinite(s) && s > 0.0 && s < 2.0; }

lb_status validate(int nx, int ny, const lb_eos *eos, double G, double kappa, double sigma,
                   const lb_rates *r, int prec, int bc, std::string &why) {
    if (nx < 3 || ny < 3) { why = "nx and ny must be >= 3"; return LB_EINVAL; }
    // the step kernel addresses a buffer with 32-bit element offsets (9 planes)
    if (9LL * (long long)lb_pitch(nx, prec) * ny >= (1LL << 32)) { why = "lattice too large"; return LB_EINVAL; }
    if (!eos || !r) { why = "eos and rates must not be NULL"; return LB_EINVAL; }
    if (prec != LB_FP32 && prec != LB_FP64 && prec != LB_BF16) {
        why = "prec must be LB_FP64, LB_FP32 or LB_BF16";
        return LB_EINVAL;
    }
    if (bc != LB_BC_PERIODIC && bc != LB_BC_WALLS_Y && bc != LB_BC_OPEN) {
        why = "bad boundary kind";
        return LB_EINVAL;
    }
    if (bc == LB_BC_OPEN && prec == LB_BF16) {
        why = "open boundaries are compiled for LB_FP32 and LB_FP64";
        return LB_EINVAL;
    }
    if (!(rate_ok(r->s_rho) && rate_ok(r->s_e) && rate_ok(r->s_zeta) && rate_ok(r->s_j) &&
          rate_ok(r->s_q) && rate_ok(r->s_v))) {
        why = "relaxation rates must lie in (0, 2) (tau > 1/2)";
        return LB_EINVAL;
    }
    if (!(std::isfinite(kappa) && kappa >= 0.0 && kappa < 1.0)) { why = "kappa must be in [0, 1)"; return LB_EINVAL; }
    if (!(std::isfinite(sigma) && sigma >= 0.0)) { why = "sigma_force must be >= 0"; return LB_EINVAL; }
    if (sigma != 0.0 && r->s_zeta != r->s_e) {
        why = "Eq. 8 requires tau_zeta == tau_e when sigma_force != 0";
        return LB_EINVAL;
    }
    if (!std::isfinite(G)) { why = "G must be finite"; return LB_EINVAL; }
    switch (eos->kind) {
        case LB_EOS_CS:
            if (!(eos->a > 0 && eos->b > 0 && eos->R > 0 && eos->T > 0)) {
                why = "Carnahan-Starling needs a, b, R, T > 0";
                return LB_EINVAL;
            }
            if (G == 0.0) { why = "G must be non-zero for the EOS-based potential"; return LB_EINVAL; }
            break;
        case LB_EOS_EXP:
            if (!(eos->psi0 > 0 && eos->rho0 > 0)) { why = "exponential potential needs psi0, rho0 > 0"; return LB_EINVAL; }
            break;
        case LB_EOS_PIECEWISE:
            if (!(eos->rho1 > 0 && eos->rho2 > eos->rho1)) { why = "Eq. 23 needs 0 < rho1 < rho2"; return LB_EINVAL; }
            if (G == 0.0) { why = "G must be non-zero for the EOS-based potential"; return LB_EINVAL; }
            break;
        default:
            why = "unknown EOS kind";
            return LB_EINVAL;
    }
    return LB_OK;
}

Consts make_consts(const lb_eos *e, double G, double kappa, double sigma, const lb_rates *r) {
    Consts c{};
    c.eos_kind = e->kind;
    c.a = e->a;
    c.b4 = e->b / 4.0;
    c.RT = e->R * e->T;
    c.psi0 = e->psi0;
    c.rho0 = e->rho0;
    c.th_v = e->theta_v;
    c.th_m = e->theta_m;
    c.th_l = e->theta_l;
    c.rho1 = e->rho1;
    c.rho2 = e->rho2;
    c.p_rho1 = e->rho1 * e->theta_v;
    c.p_rho2 = c.p_rho1 + (e->rho2 - e->rho1) * e->theta_m;
    c.two_over_G = (G != 0.0) ? 2.0 / G : 0.0;
    c.G = G;
    c.kG2 = kappa * G / 2.0;
    const double tau_e = 1.0 / r->s_e;
    c.sig_coef = 12.0 * sigma * G * G / (tau_e - 0.5);
    c.s_e = r->s_e;
    c.s_z = r->s_zeta;
    c.s_q = r->s_q;
    c.s_v = r->s_v;
    c.stall_row = INT_MIN;
    c.rho_sw = -HUGE_VAL;       // nu(rho) off
    c.s_v_vapour = c.s_v;
    return c;
}

// ---- TMA descriptors ------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// 3-D map over one population buffer: (padded column, row, population); one box is a
// lattice row of the strip plus its apron, (tx + ghost + 4) x 1 x planes: all nine
// populations for the whole-row ring, one for the stage ring (the left apron is as wide as
// the ghost offset, so a box starts at the strip's own first element), or the rows of a tile
// for the direct kernels.
lb_status encode_map(lb_ctx *c, void *buffer, CUtensorMap *map) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return fail(c, LB_ECUDA, "cuTensorMapEncodeTiled unavailable");
    const Geom &g = c->geom;
    const cuuint64_t dims[3] = {(cuuint64_t)g.pitch, (cuuint64_t)g.ny, 9};
    const cuuint64_t strides[2] = {(cuuint64_t)g.pitch * c->elem, (cuuint64_t)g.plane * c->elem};
    const bool direct = c->launch.variant >= lbm::direct_variant();
    const cuuint32_t box[3] = {
        (cuuint32_t)(direct ? lbm::TILE_BOX_W : c->launch.tx + lbm::ghost_of_prec(c->prec) + 4),
        (cuuint32_t)(direct ? lbm::TILE_BOX_ROWS : 1),
        (cuuint32_t)lbm::step_variant_planes(c->launch.variant)};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUtensorMapDataType dt = c->prec == LB_FP32   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                 : c->prec == LB_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                      : CU_TENSOR_MAP_DATA_TYPE_FLOAT64;
    CUresult r = enc(map, dt, 3, buffer, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        char buf[96];
        std::snprintf(buf, sizeof buf, "cuTensorMapEncodeTiled failed (%d)", (int)r);
        return fail(c, LB_ECUDA, buf);
    }
    return LB_OK;
}

lb_status make_maps(lb_ctx *c) {
    for (int b = 0; b < 2; ++b) {
        const lb_status s = encode_map(c, c->f[b], &c->tmap[b]);
        if (s != LB_OK) return s;
    }
    return LB_OK;
}

// whether the direct kernels can run this lattice: its rows fit a grid, and the psi scratch of
// the FP64 ones (1/18 of the two population buffers) could be allocated
bool direct_usable(lb_ctx *c) {
    if (!lbm::direct_fits(c->geom)) return false;
    if (c->prec != LB_FP64 || c->d_psi) return true;
    if (cudaMalloc(&c->d_psi, (size_t)c->geom.plane * c->elem) == cudaSuccess) return true;
    (void)cudaGetLastError();
    c->d_psi = nullptr;
    return false;
}

// which kernel takes several steps of this lattice in one launch, see lb_ctx::many
int many_usable(lb_ctx *c) {
    if (lbm::cluster_fits(c->prec, c->consts, c->geom)) return 1;
    const size_t bytes = lbm::resident_bytes(c->prec, c->consts, c->geom, c->num_sms);
    if (bytes == 0) return 0;
    if (c->d_words) return 2;
    if (cudaMalloc(&c->d_words, bytes) == cudaSuccess &&
        cudaMemsetAsync(c->d_words, 0, bytes, c->stream) == cudaSuccess)
        return 2;
    (void)cudaGetLastError();
    cudaFree(c->d_words);
    c->d_words = nullptr;
    return 0;
}

// any_many: several steps go together with any variant, not only with the one that contexts start with
lb_status apply_launch(lb_ctx *c, int variant, int rows, bool any_many = false) {
    if (variant < 0 || variant >= lbm::step_variant_count())
        return fail(c, LB_EINVAL, "unknown launch variant");
    if (rows < 0) return fail(c, LB_EINVAL, "rows must be >= 0");
    c->asked_variant = variant;
    c->asked_rows = rows;
    c->asked_many = any_many;
    if (variant >= lbm::direct_variant()) {
        if (c->prec == LB_FP64) variant = lbm::direct_variant();     // no staged FP64 kernel
        if (!direct_usable(c)) variant = lbm::default_ring_variant();
    }
    c->many = any_many || variant == lbm::default_variant(c->prec, c->geom) ? many_usable(c) : 0;
    const int stall = c->consts.stall_row;
    if (stall != INT_MIN) {      // test hook: kernels that wait for the row
        if (c->many == 1 || !lbm::resident_waits_for_row(c->geom, stall)) c->many = 0;
        if (variant == lbm::direct_variant() ||
            (variant == lbm::staged_variant() && !lbm::staged_loads_row(c->geom, stall)))
            variant = lbm::default_ring_variant();
    }
    c->launch = lbm::make_step_launch(c->prec, c->consts.eos_kind, c->geom, c->num_sms, variant, rows);
    LB_CUDA(c, lbm::configure_step(c->prec, c->consts, c->geom, c->launch));
    return variant >= lbm::direct_variant() && c->prec == LB_FP64 ? LB_OK : make_maps(c);
}

// a launch of many steps that the GPU (or this process's share of it) has no room for: the steps can
// still be taken one by one. Any other error is the caller's to know.
bool no_room(cudaError_t e) {
    return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorInvalidClusterSize ||
           e == cudaErrorLaunchOutOfResources || e == cudaErrorInvalidConfiguration;
}

lb_status check_usable(lb_ctx *c) {
    if (!c) return LB_EINVAL;
    return c->sticky;
}

// Wait for the stream and fold device error bits into the sticky status. The kernels write them
// (and a reduction's results) into host memory, so there is nothing to copy: a wait
// and a blocking copy of the error word took 14 us, the wait alone takes 5.
lb_status sync_and_check(lb_ctx *c) {
    LB_CUDA(c, cudaStreamSynchronize(c->stream));
    const int flags = *static_cast<volatile int *>(&c->words->err);
    if (flags & lbm::ERR_TIMEOUT)
        return poison(c, LB_ETIMEOUT, "a bounded device-side wait gave up");
    if (flags & lbm::ERR_DOMAIN)
        return poison(c, LB_EDOMAIN, "psi^2 < 0 or rho <= 0 at some site (EOS domain left)");
    return LB_OK;
}

// The words that the kernels write and the host reads. Where the GPU reads the host's page tables
// (GB300) they are ordinary memory: a page-locked allocation and its release take 270 us, which made
// lb_init and lb_free of a 64^2 lattice 560 us (55 now).
cudaError_t make_words(lb_ctx *c, int dev) {
    constexpr size_t line = 128;         // whole cache lines, nothing else in them
    static_assert(sizeof(lbm::HostWords) <= line, "one line");
    int host_tables = 0;
    cudaError_t e = cudaDeviceGetAttribute(&host_tables, cudaDevAttrPageableMemoryAccessUsesHostPageTables, dev);
    if (e != cudaSuccess) return e;
    void *host = nullptr, *device = nullptr;
    if (host_tables) {
        host = device = std::aligned_alloc(line, line);
        if (!host) return cudaErrorMemoryAllocation;
    } else {
        e = cudaHostAlloc(&host, line, cudaHostAllocMapped);
        c->words_locked = e == cudaSuccess;
    }
    c->words = static_cast<lbm::HostWords *>(host);
    if (e == cudaSuccess && !host_tables) e = cudaHostGetDevicePointer(&device, host, 0);
    if (e != cudaSuccess) return e;
    std::memset(host, 0, line);
    c->d_err = &static_cast<lbm::HostWords *>(device)->err;
    c->d_out8 = static_cast<lbm::HostWords *>(device)->out8;
    return cudaSuccess;
}

lb_status ensure_diag(lb_ctx *c) {
    const size_t n = (size_t)c->geom.nx * c->geom.ny;
    if (!c->d_field) LB_CUDA(c, cudaMalloc(&c->d_field, 2 * n * sizeof(double)));
    if (!c->d_partials) {
        const size_t k = 8 * (size_t)lbm::reduce_blocks((long long)n);
        double *partials = nullptr;
        LB_CUDA(c, cudaMalloc(&partials, (k + 1) * sizeof(double)));
        const cudaError_t e = cudaMemsetAsync(partials + k, 0, sizeof(double), c->stream);
        if (e != cudaSuccess) cudaFree(partials);
        LB_CUDA(c, e);
        c->d_partials = partials;
        c->d_ticket = reinterpret_cast<unsigned *>(partials + k);
    }
    if (!c->d_first) LB_CUDA(c, cudaMalloc(&c->d_first, sizeof(int) * (size_t)c->geom.nx));
    return LB_OK;
}

void *spare(lb_ctx *c) { return c->f[c->cur ^ 1]; }

lb_status create(lb_ctx **out, int nx, int ny, const lb_eos *eos, double G, double kappa,
                 double sigma, const lb_rates *rates, int prec, int bc, void *stream, void *fa,
                 void *fb, bool external) {
    if (!out) return LB_EINVAL;
    *out = nullptr;
    std::string why;
    lb_status s = validate(nx, ny, eos, G, kappa, sigma, rates, prec, bc, why);
    if (s != LB_OK) {
        std::fprintf(stderr, "lb_init: %s\n", why.c_str());
        return s;
    }
    if (external) {
        if (!fa || !fb || fa == fb) return LB_EINVAL;
        if ((reinterpret_cast<uintptr_t>(fa) | reinterpret_cast<uintptr_t>(fb)) & 255u) return LB_EINVAL;
    }
    lb_ctx *c = new (std::nothrow) lb_ctx();
    if (!c) return LB_ENOMEM;
    c->prec = prec;
    c->elem = elem_size(prec);
    c->geom.nx = nx;
    c->geom.ny = ny;
    c->geom.pitch = (int)lb_pitch(nx, prec);
    c->geom.plane = (long long)ny * c->geom.pitch;
    c->geom.walls = bc;   // the boundary kind
    c->consts = make_consts(eos, G, kappa, sigma, rates);
    c->stream = static_cast<cudaStream_t>(stream);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) {
        std::fprintf(stderr, "lb_init: %s\n", cudaGetErrorString(e));
        delete c;
        return lbm::reported(LB_ECUDA);
    }
    const size_t bytes = lb_buffer_bytes(nx, ny, prec);
    if (external) {
        c->f[0] = fa;
        c->f[1] = fb;
        c->own_f = false;
    } else {
        c->own_f = true;
        if (cudaMalloc(&c->f[0], bytes) != cudaSuccess || cudaMalloc(&c->f[1], bytes) != cudaSuccess) {
            lb_free(c);
            return lbm::reported(LB_ENOMEM);
        }
    }
    if (make_words(c, dev) != cudaSuccess) {
        lb_free(c);
        return lbm::reported(LB_ENOMEM);
    }
    if (cudaMemsetAsync(c->f[0], 0, bytes, c->stream) != cudaSuccess ||
        cudaMemsetAsync(c->f[1], 0, bytes, c->stream) != cudaSuccess ||
        cudaStreamSynchronize(c->stream) != cudaSuccess) {
        lb_free(c);
        return lbm::reported(LB_ECUDA);
    }
    if ((s = apply_launch(c, lbm::default_variant(prec, c->geom), 0)) != LB_OK) {
        std::fprintf(stderr, "lb_init: %s\n", c->msg.c_str());
        lb_free(c);
        return lbm::reported(s);
    }
    *out = c;
    return LB_OK;
}

}  // namespace

namespace lbm {

lb_status ctx_view(const lb_ctx *c, CtxView *v) {
    if (!c || !v) return LB_EINVAL;
    v->g = c->f[c->cur];
    v->geom = c->geom;
    v->consts = c->consts;
    v->prec = c->prec;
    v->stream = c->stream;
    v->sticky = c->sticky;
    return LB_OK;
}

lb_status ctx_fail(lb_ctx *c, lb_status s, const char *msg, bool poison_ctx) {
    if (!c) return s;
    c->msg = msg ? msg : "";
    if (poison_ctx) c->sticky = s;
    return reported(s);
}

lb_status ctx_sync_check(lb_ctx *c) {
    if (!c) return LB_EINVAL;
    return sync_and_check(c);
}

}  // namespace lbm

extern "C" {

size_t lb_pitch(int nx, int prec) {
    (void)prec;
    if (nx <= 0) return 0;
    return (size_t)((nx + 2 * lbm::ghost_of_prec(prec) + 31) / 32) * 32;
}

size_t lb_buffer_bytes(int nx, int ny, int prec) {
    if (nx <= 0 || ny <= 0) return 0;
    return 9 * (size_t)ny * lb_pitch(nx, prec) * elem_size(prec);
}

lb_status lb_init(lb_ctx **out, int nx, int ny, const lb_eos *eos, double G, double kappa,
                  double sigma_force, const lb_rates *rates, int prec, int bc, void *stream) {
    return create(out, nx, ny, eos, G, kappa, sigma_force, rates, prec, bc, stream, nullptr,
                  nullptr, false);
}

lb_status lb_init_ex(lb_ctx **out, int nx, int ny, const lb_eos *eos, double G, double kappa,
                     double sigma_force, const lb_rates *rates, int prec, int bc, void *stream,
                     void *f_a, void *f_b) {
    return create(out, nx, ny, eos, G, kappa, sigma_force, rates, prec, bc, stream, f_a, f_b,
                  true);
}

int lb_launch_variants(void) { return lbm::step_variant_count(); }

lb_status lb_set_launch(lb_ctx *c, int variant, int rows) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    LB_CUDA(c, cudaStreamSynchronize(c->stream));
    return apply_launch(c, variant, rows);
}

lb_status lb_autotune(lb_ctx *c, int trial_steps, int *variant, int *rows) {
    const lbm::NvtxRange nvtx_range("lb_autotune");
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (trial_steps < 1) return fail(c, LB_EINVAL, "lb_autotune: trial_steps < 1");
    // device errors of earlier steps are the state's: report them before any trial
    if ((s = sync_and_check(c)) != LB_OK) return s;
    // Launches of many steps beat all that could be tried here: what is chosen is the launch of single
    // steps, between the two tile kernels (the ring kernels take twice their time and more at these sizes).
    const bool many = many_usable(c) != 0;
    static const int cand[] = {0, 6, 8, 9, 10, 11, 12, 13, 14, 15, 16, 20, 24};
    // Trial launches take real steps on a scratch copy of the state, ping-ponging with the
    // spare buffer as lb_step does (each launch reads what the previous one wrote, in the
    // alternating visiting order), so every candidate meets the L2 reuse of real stepping;
    // the state itself is only read. Without room for the copy, every trial reads the
    // state and writes the spare buffer instead.
    const size_t bytes = lb_buffer_bytes(c->geom.nx, c->geom.ny, c->prec);
    void *scratch = nullptr;
    if (cudaMalloc(&scratch, bytes) != cudaSuccess) {
        (void)cudaGetLastError();
        scratch = nullptr;
    } else if (cudaMemcpyAsync(scratch, c->f[c->cur], bytes, cudaMemcpyDeviceToDevice,
                               c->stream) != cudaSuccess) {
        cudaFree(scratch);
        return fail(c, LB_ECUDA, "lb_autotune: copy of the state failed");
    }
    CUtensorMap scratch_map;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        if (scratch) cudaFree(scratch);
        return fail(c, LB_ECUDA, "lb_autotune: cudaEventCreate failed");
    }
    float best_ms = 0.f;
    int best_v = c->launch.variant, best_r = c->launch.rows;
    cudaError_t e = cudaSuccess;
    for (int v = 0; v < lbm::step_variant_count() && e == cudaSuccess; ++v) {
        int tried_rows[16], n_tried = 0;
        const bool direct = v >= lbm::direct_variant();
        if (many && !direct) continue;
        if (direct && !direct_usable(c)) continue;
        if (v == lbm::staged_variant() && c->prec == LB_FP64) continue;
        for (int r : cand) {
            if (direct && r != 0) break;      // one launch shape
            if ((s = apply_launch(c, v, r)) != LB_OK) break;
            const int rr = c->launch.rows;
            bool seen = false;
            for (int i = 0; i < n_tried; ++i) seen |= tried_rows[i] == rr;
            if (seen) continue;
            tried_rows[n_tried++] = rr;
            if (scratch && !(direct && c->prec == LB_FP64) && (s = encode_map(c, scratch, &scratch_map)) != LB_OK) break;
            // trial k reads the scratch copy (k even) or the spare buffer (k odd) and
            // writes the other, in visiting order k & 1
            int k = 0;
            auto once = [&]() {
                const bool from_scratch = (k & 1) == 0;
                lbm::StepBuffers b;
                b.tensor_map_in = !scratch       ? &c->tmap[c->cur]
                                  : from_scratch ? &scratch_map
                                                 : &c->tmap[c->cur ^ 1];
                b.gin = !scratch ? c->f[c->cur] : from_scratch ? scratch : c->f[c->cur ^ 1];
                b.gout = (!scratch || from_scratch) ? c->f[c->cur ^ 1] : scratch;
                b.psi = c->d_psi;
                const cudaError_t r = lbm::launch_step(c->prec, c->consts, c->geom, c->launch,
                                                       k & 1, b, c->d_err, c->stream);
                ++k;
                return r;
            };
            e = once();
            // best of three timed runs: a single short run is at the mercy of clock and
            // memory-controller noise of a few percent, the size of the differences sought
            float ms = 0.f;
            for (int rep = 0; rep < 3 && e == cudaSuccess; ++rep) {
                e = cudaEventRecord(e0, c->stream);
                for (int i = 0; i < trial_steps && e == cudaSuccess; ++i) e = once();
                if (e == cudaSuccess) e = cudaEventRecord(e1, c->stream);
                if (e == cudaSuccess) e = cudaEventSynchronize(e1);
                float t = 0.f;
                if (e == cudaSuccess) e = cudaEventElapsedTime(&t, e0, e1);
                if (e == cudaSuccess && (rep == 0 || t < ms)) ms = t;
            }
            if (e != cudaSuccess) break;
            if (best_ms == 0.f || ms < best_ms) {
                best_ms = ms;
                best_v = v;
                best_r = rr;
            }
        }
        if (s != LB_OK) break;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (scratch) cudaFree(scratch);
    if (s != LB_OK) return s;
    if (e != cudaSuccess)
        return fail(c, LB_ECUDA, std::string("lb_autotune: ") + cudaGetErrorString(e));
    // the trials stepped a copy: a domain error there says nothing about the state; a
    // timeout (a bounded wait gave up) is kept, it concerns the kernel and not the data
    if (c->words->err & lbm::ERR_TIMEOUT)       // (the stream has been waited for)
        return poison(c, LB_ETIMEOUT, "a bounded device-side wait gave up");
    c->words->err = 0;
    if ((s = apply_launch(c, best_v, best_r, many)) != LB_OK) return s;
    if (variant) *variant = best_v;
    if (rows) *rows = best_r;
    return sync_and_check(c);
}

lb_status lb_set_viscosity_switch(lb_ctx *c, double rho_1, double s_v_vapour) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (c->geom.walls != LB_BC_OPEN)
        return fail(c, LB_EINVAL, "lb_set_viscosity_switch: LB_BC_OPEN contexts only");
    if (!(std::isfinite(rho_1) && rate_ok(s_v_vapour)))
        return fail(c, LB_EINVAL, "lb_set_viscosity_switch: need a finite rho_1 and s_v in (0, 2)");
    LB_CUDA(c, cudaStreamSynchronize(c->stream));
    c->consts.rho_sw = rho_1;
    c->consts.s_v_vapour = s_v_vapour;
    return LB_OK;
}

lb_status lb_set_storage_shift(lb_ctx *c, double rho_s) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (c->prec != LB_BF16) return fail(c, LB_EINVAL, "lb_set_storage_shift: LB_BF16 contexts only");
    if (!std::isfinite(rho_s)) return fail(c, LB_EINVAL, "lb_set_storage_shift: non-finite rho_s");
    LB_CUDA(c, cudaStreamSynchronize(c->stream));
    c->consts.shift_rho = rho_s;
    return LB_OK;
}

lb_status lb_set_storage_rounding(lb_ctx *c, int mode) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (c->prec != LB_BF16) return fail(c, LB_EINVAL, "lb_set_storage_rounding: LB_BF16 contexts only");
    if (mode != LB_ROUND_NEAREST && mode != LB_ROUND_STOCHASTIC)
        return fail(c, LB_EINVAL, "lb_set_storage_rounding: unknown mode");
    LB_CUDA(c, cudaStreamSynchronize(c->stream));
    c->consts.stochastic = mode == LB_ROUND_STOCHASTIC ? 1 : 0;
    return LB_OK;
}

lb_status lb_debug_stall_row(lb_ctx *c, int row) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    c->consts.stall_row = row;
    return apply_launch(c, c->asked_variant, c->asked_rows, c->asked_many);
}

lb_status lb_get_launch(const lb_ctx *c, int *variant, int *tx, int *rows, int *ctas_per_sm) {
    if (!c) return LB_EINVAL;
    if (variant) *variant = c->launch.variant;
    if (tx) *tx = c->launch.tx;
    if (rows) *rows = c->launch.rows;
    if (ctas_per_sm)
        *ctas_per_sm = c->launch.variant >= lbm::direct_variant()
                           ? lbm::tile_occupancy(c->prec, c->consts, c->geom, c->launch.variant)
                           : c->launch.ctas_per_sm;
    return LB_OK;
}

lb_status lb_set_rho_u(lb_ctx *c, const double *rho, const double *ux, const double *uy) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (!rho || !ux || !uy) return fail(c, LB_EINVAL, "lb_set_rho_u: NULL array");
    const size_t n = (size_t)c->geom.nx * c->geom.ny;
    if (!c->d_host_in) LB_CUDA(c, cudaMalloc(&c->d_host_in, 3 * n * sizeof(double)));
    LB_CUDA(c, cudaMemcpyAsync(c->d_host_in, rho, n * sizeof(double), cudaMemcpyHostToDevice, c->stream));
    LB_CUDA(c, cudaMemcpyAsync(c->d_host_in + n, ux, n * sizeof(double), cudaMemcpyHostToDevice, c->stream));
    LB_CUDA(c, cudaMemcpyAsync(c->d_host_in + 2 * n, uy, n * sizeof(double), cudaMemcpyHostToDevice, c->stream));
    LB_CUDA(c, lbm::launch_init_feq(c->prec, c->consts, c->geom, c->d_host_in, c->d_host_in + n,
                                    c->d_host_in + 2 * n, spare(c), c->d_err, c->stream));
    LB_CUDA(c, lbm::launch_unstream(c->prec, c->geom, spare(c), c->f[c->cur], false, c->stream));
    c->steps = 0;
    return sync_and_check(c);
}

lb_status lb_step(lb_ctx *c, int n) {
    const lbm::NvtxRange nvtx_range("lb_step");
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (n < 0) return fail(c, LB_EINVAL, "lb_step: n < 0");
    // a lattice that fits the SMs takes several steps in one launch (at most kManySteps: a few
    // milliseconds)
    while (c->many && n >= kManyLeast[c->many]) {
        const int m = std::min(n, kManySteps);
        const void *gin = c->f[c->cur];
        void *gout = c->f[c->cur ^ (m & 1)];     // the buffer that m launches would end in
        const cudaError_t e =
            c->many == 1 ? lbm::launch_cluster_steps(c->consts, c->geom, gin, gout, m, c->d_err, c->stream)
                         : lbm::launch_resident_steps(c->consts, c->geom, c->num_sms, gin, gout, m, c->d_words,
                                                      c->d_err, c->stream);
        if (no_room(e)) {             // not every SM can be had (a limited context): single launches
            (void)cudaGetLastError();
            c->many = 0;
            break;
        }
        LB_CUDA(c, e);
        c->cur ^= m & 1;
        c->steps += m;
        ++c->launches;
        n -= m;
    }
    for (int i = 0; i < n; ++i) {
        // alternate the visiting order: each step first reads the rows the previous one
        // wrote last (still in L2 when the state is not much larger than L2)
        c->consts.step_key = (unsigned)c->steps;   // the stochastic-rounding counter
        const lbm::StepBuffers b{c->f[c->cur], &c->tmap[c->cur], c->f[c->cur ^ 1], c->d_psi};
        LB_CUDA(c, lbm::launch_step(c->prec, c->consts, c->geom, c->launch, (int)(c->steps & 1),
                                    b, c->d_err, c->stream));
        c->cur ^= 1;
        ++c->steps;
        c->launches += lb_kernels_per_step(c);
    }
    return LB_OK;
}

lb_status lb_sync(lb_ctx *c) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    return sync_and_check(c);
}

lb_status lb_get_rho(lb_ctx *c, double *rho) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (!rho) return fail(c, LB_EINVAL, "lb_get_rho: NULL");
    if ((s = ensure_diag(c)) != LB_OK) return s;
    const size_t n = (size_t)c->geom.nx * c->geom.ny;
    LB_CUDA(c, lbm::launch_macro_fields(c->prec, c->consts, c->geom, c->f[c->cur], nullptr,
                                        c->d_field, nullptr, nullptr, c->stream));
    LB_CUDA(c, cudaMemcpyAsync(rho, c->d_field, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    return sync_and_check(c);
}

lb_status lb_get_u(lb_ctx *c, double *ux, double *uy) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (!ux || !uy) return fail(c, LB_EINVAL, "lb_get_u: NULL");
    if ((s = ensure_diag(c)) != LB_OK) return s;
    const size_t n = (size_t)c->geom.nx * c->geom.ny;
    // psi goes into the spare population buffer (free between steps)
    LB_CUDA(c, lbm::launch_psi_field(c->prec, c->consts, c->geom, c->f[c->cur], spare(c),
                                     c->d_err, c->stream));
    LB_CUDA(c, lbm::launch_macro_fields(c->prec, c->consts, c->geom, c->f[c->cur], spare(c),
                                        nullptr, c->d_field, c->d_field + n, c->stream));
    LB_CUDA(c, cudaMemcpyAsync(ux, c->d_field, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    LB_CUDA(c, cudaMemcpyAsync(uy, c->d_field + n, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    return sync_and_check(c);
}

lb_status lb_get_populations(lb_ctx *c, void *dst, size_t bytes) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    const size_t row = (size_t)c->geom.nx * c->elem;
    if (!dst || bytes != 9 * (size_t)c->geom.ny * row)
        return fail(c, LB_EINVAL, "lb_get_populations: NULL or size mismatch");
    // pull into the spare buffer in the host layout, then one contiguous copy
    LB_CUDA(c, lbm::launch_stream(c->prec, c->geom, c->f[c->cur], spare(c), true, c->stream));
    LB_CUDA(c, cudaMemcpyAsync(dst, spare(c), bytes, cudaMemcpyDeviceToHost, c->stream));
    return sync_and_check(c);
}

lb_status lb_set_populations(lb_ctx *c, const void *src, size_t bytes) {
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    const size_t row = (size_t)c->geom.nx * c->elem;
    if (!src || bytes != 9 * (size_t)c->geom.ny * row)
        return fail(c, LB_EINVAL, "lb_set_populations: NULL or size mismatch");
    // one contiguous copy into the spare buffer (host layout), then the kernel unpacks it
    LB_CUDA(c, cudaMemcpyAsync(spare(c), src, bytes, cudaMemcpyHostToDevice, c->stream));
    LB_CUDA(c, lbm::launch_unstream(c->prec, c->geom, spare(c), c->f[c->cur], true, c->stream));
    return sync_and_check(c);
}

lb_status lb_reduce(lb_ctx *c, double out[4]) {
    const lbm::NvtxRange nvtx_range("lb_reduce");
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (!out) return fail(c, LB_EINVAL, "lb_reduce: NULL");
    if ((s = ensure_diag(c)) != LB_OK) return s;
    LB_CUDA(c, lbm::launch_psi_field(c->prec, c->consts, c->geom, c->f[c->cur], spare(c),
                                     c->d_err, c->stream));
    LB_CUDA(c, lbm::launch_macro_reduce(c->prec, c->consts, c->geom, c->f[c->cur], spare(c),
                                        c->d_partials, c->d_ticket, c->d_out8, c->stream));
    s = sync_and_check(c);
    for (int i = 0; i < 3; ++i) out[i] = c->words->out8[i];
    out[3] = std::sqrt(c->words->out8[3]);   // the reduction's maximum is of |v|^2
    if (s != LB_OK) return s;
    for (int i = 0; i < 4; ++i)
        if (!std::isfinite(out[i]))
            return poison(c, LB_ENONFINITE, "lb_reduce: non-finite mass, momentum or |v|");
    return LB_OK;
}

lb_status lb_measure_droplet(lb_ctx *c, double radius, double out[8]) {
    const lbm::NvtxRange nvtx_range("lb_measure_droplet");
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (!out) return fail(c, LB_EINVAL, "lb_measure_droplet: NULL");
    if (!(radius > 0 && std::isfinite(radius)))
        return fail(c, LB_EINVAL, "lb_measure_droplet: radius must be positive and finite");
    if ((s = ensure_diag(c)) != LB_OK) return s;
    const int nx = c->geom.nx, ny = c->geom.ny;
    const double r_out = radius + 0.3 * 0.5 * std::min(nx, ny);
    LB_CUDA(c, lbm::launch_droplet_sums(c->prec, c->consts, c->geom, c->f[c->cur], 0.5 * radius,
                                        r_out, c->d_partials, c->d_ticket, c->d_out8, c->stream));
    if ((s = sync_and_check(c)) != LB_OK) return s;
    lbm::droplet_results(c->words->out8, (double)nx * ny, false, out);
    return LB_OK;
}

lb_status lb_interface_height(lb_ctx *c, double rho_mid, double *heights) {
    const lbm::NvtxRange nvtx_range("lb_interface_height");
    lb_status s = check_usable(c);
    if (s != LB_OK) return s;
    if (!heights) return fail(c, LB_EINVAL, "lb_interface_height: NULL");
    if (!std::isfinite(rho_mid)) return fail(c, LB_EINVAL, "lb_interface_height: non-finite rho_mid");
    if ((s = ensure_diag(c)) != LB_OK) return s;
    LB_CUDA(c, lbm::launch_interface_height(c->prec, c->consts, c->geom, c->f[c->cur], rho_mid,
                                            c->d_first, c->d_field, c->stream));
    LB_CUDA(c, cudaMemcpyAsync(heights, c->d_field, sizeof(double) * (size_t)c->geom.nx,
                               cudaMemcpyDeviceToHost, c->stream));
    return sync_and_check(c);
}

long long lb_steps_done(const lb_ctx *c) { return c ? c->steps : 0; }

long long lb_step_launches(const lb_ctx *c) { return c ? c->launches : 0; }

int lb_kernels_per_step(const lb_ctx *c) {
    if (!c) return 0;
    return c->prec == LB_FP64 && c->launch.variant == lbm::direct_variant() ? 2 : 1;
}

const char *lb_last_error(const lb_ctx *c) { return c ? c->msg.c_str() : kNoCtx; }

lb_status lb_status_of(const lb_ctx *c) { return c ? c->sticky : LB_EINVAL; }

void lb_free(lb_ctx *c) {
    if (!c) return;
    if (c->stream) cudaStreamSynchronize(c->stream);
    else cudaDeviceSynchronize();
    if (c->own_f) {
        cudaFree(c->f[0]);
        cudaFree(c->f[1]);
    }
    cudaFree(c->d_field);
    cudaFree(c->d_partials);
    cudaFree(c->d_first);
    cudaFree(c->d_host_in);
    cudaFree(c->d_psi);
    cudaFree(c->d_words);
    // as cudaFree does, for what other streams (replayed captures) may still write there
    if (c->words) cudaDeviceSynchronize();
    if (c->words_locked) cudaFreeHost(c->words);
    else std::free(c->words);
    delete c;
}

}  // extern "C"
