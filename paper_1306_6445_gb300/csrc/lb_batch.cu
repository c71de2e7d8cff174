// Batched lattices (lb_batch_*): many independent periodic droplet lattices of uneven size
// and parameters advanced together, plus per-lattice Laplace measurements on the GPU. FP32 batches
// take their steps by groups of lattices whose state stays in L2 (k_batch_tile, queue_groups); FP64
// and the ring variants by one persistent kernel per time step over all lattices (k_batch_step),
// replayed from a captured CUDA graph. Steps of the groups are graphs too (launch_graphs).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "lb_device.cuh"
#include "lb_internal.h"

namespace {

constexpr int kGraphSteps = 64;   // steps per captured graph (even: the phase returns)
// Several groups: graphs of 64 steps of up to 8 groups, 32 of up to 16, 16 of more, in blocks of 48
// groups. lb_batch_step can return without waiting only if it queues few operations: launched one by
// one, 64 steps of 512 lattices of 64^2 to 512^2 (229 groups) hold the calling thread for 30 of their
// 39.1 ms, of 24 x 128^2 (3 groups) for 0.39 of 0.40 ms; as graphs 0.1 of 39.25 ms and 0.004 of 0.33. The
// shorter the graphs, the more the groups' states are read again and the chains started and drained
// (24 x 128^2: 16 steps 359 us; the 512 lattices: 32 steps 38.7 ms, blocks of 24 or 12 groups 39.6 and
// 40.7), the longer, the longer they take to make: 4 us per group and step (15 ms for the 512
// lattices, during which the GPU takes the steps of the blocks before). So the first 512 steps of a
// batch, and after its launch or active lattices have changed, are launched one by one.
constexpr size_t kBlockGroups = 48;
constexpr int kDirectSteps = 512;
// Most sites of a group of the staged tiles (or one lattice): both buffers of the kChains groups
// that run side by side (57 MB in FP32) stay in L2 over their steps. 64 steps of 512 lattices of
// 64^2 to 512^2, sites / groups side by side: 2^18 / 3 39.4 ms, 2^18 / 2 45.8, 2^18 / 4 41.4, 0.7 2^18
// / 3 40.4, 1.4 2^18 / 3 41.0, 2^19 / 2 40.4, 2^20 / 1 51.7; of 512 lattices of 128^2: 6.7, 6.8, 8.6,
// 6.6, 8.5, 7.8, 9.2. All lattices in one launch of the ring kernel: 50.2 ms.
constexpr long long kGroupSites = 1 << 18;
constexpr long long kShortSites = 1 << 17;   // a smaller batch is one group (and one graph)
constexpr int kChains = 3;        // groups that run side by side, see queue_groups

struct BatchCommon {
    int n = 0;
    int prec = LB_FP32;
    int eos_kind = LB_EOS_CS;
    size_t elem = 4;
    cudaStream_t stream = nullptr;
    std::vector<lbm::Geom> geom;
    std::vector<lbm::Consts> consts;
    std::vector<size_t> off[2];          // byte offsets of each lattice's two buffers
    void *pool = nullptr;                // all population buffers
    void *d_maps = nullptr;              // 2 CUtensorMap per lattice, of the staged tiles
    void *d_lats = nullptr;              // BatchLattice<T> table
    // A ring variant's launch: all lattices, one step. `ring` is the batch's where its variant is one;
    // `few` takes the calls of up to few_steps steps beside the staged tiles (lb_batch_autotune).
    struct Ring {
        int variant = 0, rows = 0, grid = 0, n_items = 0;
        lbm::BatchItem *d_items = nullptr;
        void *d_maps = nullptr;          // 2 CUtensorMap per lattice
    } ring, few;
    int few_steps = 0;
    int n_items = 0;
    // Lattices that take their steps together (lb_batch_step): the staged tiles (variant 8) have
    // groups that stay in L2, the ring variants one group of all items.
    struct Group {
        lbm::BatchGroup lattices{};      // staged tiles: the lattices, how many, most tiles of one
        int n = 0, max_tiles = 0;
    };
    std::vector<Group> groups;
    cudaStream_t side[kChains - 1] = {};             // see queue_groups
    cudaEvent_t fork = nullptr, join[kChains - 1] = {};
    int *d_errs = nullptr;
    double *d_stage = nullptr;           // rho, ux, uy staging for one lattice
    size_t stage_sites = 0;
    double *d_radius = nullptr;
    double *d_meas = nullptr;
    lbm::MeasureChunk *d_chunks = nullptr;   // CTAs of a measurement (all lattices)
    int *d_first = nullptr;                  // first chunk of lattice i, n + 1 entries
    double *d_partials = nullptr;            // 8 doubles per chunk
    int n_chunks = 0;
    int *h_errs = nullptr;                   // page-locked: error words, radii, measured sums
    double *h_radius = nullptr, *h_meas = nullptr;
    int variant = 0, rows = 16, grid = 0, num_sms = 0;
    int phase = 0;                       // which buffer holds the active lattices' state
    std::vector<unsigned char> active;   // lattices stepped by lb_batch_step
    std::vector<long long> lat_steps;    // steps taken by each lattice
    long long steps = 0;
    // graph_steps steps of each block of kBlockGroups groups from phase 0 / 1
    std::vector<cudaGraphExec_t> graphs[2];
    int direct_steps = 0;                // launched one by one since the groups were formed
    bool no_graphs = false;              // one could not be made
    long long queued = 0;                // launches of steps, also of graphs of them
    lb_status sticky = LB_OK;
    std::string msg;
};

}  // namespace

struct lb_batch : BatchCommon {};

namespace {

lb_status bfail(lb_batch *b, lb_status s, const std::string &m, bool poison = false) {
    if (b) {
        b->msg = m;
        if (poison) b->sticky = s;
    }
    return lbm::reported(s);
}

#define LB_BCUDA(b, call)                                                            \
    do {                                                                             \
        cudaError_t e__ = (call);                                                    \
        if (e__ != cudaSuccess)                                                      \
            return bfail(b, LB_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e__)); \
    } while (0)

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn batch_encode_fn() {
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

void *buf(lb_batch *b, int i, int which) {
    return static_cast<char *>(b->pool) + b->off[which][i];
}

// Work items for a strip width `tx` and `rows` rows per item: each lattice is cut into
// ceil(nx / tx) strips (lb_strip_widths) and row blocks of `rows` rows marching
// alternately up and down; items are ordered lattice by lattice so that the neighbours of
// a row block run at the same time. Every strip starts on a multiple of 4 columns (the
// TMA start coordinate must be 16-byte aligned); an item that would not is refused.
bool make_items(const lb_batch *b, int tx, int rows, std::vector<lbm::BatchItem> &items) {
    items.clear();
    std::vector<int> widths(4096);
    for (int i = 0; i < b->n; ++i) {
        if (!b->active[i]) continue;     // an inactive lattice has no work items
        const int nx = b->geom[i].nx, ny = b->geom[i].ny;
        const int ns = lb_strip_widths(nx, tx, widths.data(), (int)widths.size());
        if (ns <= 0) return false;
        const int nb = (ny + rows - 1) / rows;
        for (int rb = 0; rb < nb; ++rb) {
            int x0 = 0;
            for (int k = 0; k < ns; ++k) {
                lbm::BatchItem it;
                it.lat = i;
                it.x0 = x0;
                it.w = widths[k];
                it.yb = rb * rows;
                it.n = std::min(rows, ny - it.yb);
                it.dir = (rb & 1) ? -1 : 1;
                if ((it.x0 & 3) != 0 || it.w < 1 || it.w > tx || it.x0 + it.w > nx || it.n < 1)
                    return false;
                items.push_back(it);
                x0 += widths[k];
            }
        }
    }
    return true;
}

// The chunks of a measurement: whole rows, 8192 sites each (32 per thread) or, in a small batch,
// as few as 1024, so that the SMs have four CTAs each; at most 256 per lattice (one pass of
// k_batch_measure_sum's lanes over eight).
lb_status make_chunks(lb_batch *b) {
    long long all = 0;
    for (const auto &g : b->geom) all += (long long)g.nx * g.ny;
    const int sites = (int)std::max<long long>(1024, std::min<long long>(8192, all / (4 * b->num_sms)));
    std::vector<lbm::MeasureChunk> chunks;
    std::vector<int> first(b->n + 1);
    for (int i = 0; i < b->n; ++i) {
        first[i] = (int)chunks.size();
        const int nx = b->geom[i].nx, ny = b->geom[i].ny;
        const int rows = std::max(std::max(1, sites / nx), (ny + 255) / 256);
        for (int y = 0; y < ny; y += rows) chunks.push_back({i, y, std::min(rows, ny - y)});
    }
    first[b->n] = b->n_chunks = (int)chunks.size();
    if (cudaMalloc(&b->d_chunks, chunks.size() * sizeof(chunks[0])) != cudaSuccess ||
        cudaMalloc(&b->d_first, first.size() * sizeof(int)) != cudaSuccess ||
        cudaMalloc(&b->d_partials, chunks.size() * 8 * sizeof(double)) != cudaSuccess) {
        (void)cudaGetLastError();
        return LB_ENOMEM;
    }
    if (cudaMemcpy(b->d_chunks, chunks.data(), chunks.size() * sizeof(chunks[0]),
                   cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->d_first, first.data(), first.size() * sizeof(int),
                   cudaMemcpyHostToDevice) != cudaSuccess)
        return LB_ECUDA;
    return LB_OK;
}

// The groups of the staged tiles: active lattices by size (so that the lattices of a group have
// about as many tiles), each group of at most kGroupSites sites (or one lattice) and of at most
// GROUP_LATTICES lattices. Returns the number of tiles.
int make_groups(lb_batch *b) {
    b->groups.clear();
    std::vector<int> order;
    for (int i = 0; i < b->n; ++i)
        if (b->active[i]) order.push_back(i);
    auto sites = [&](int i) { return (long long)b->geom[i].nx * b->geom[i].ny; };
    std::stable_sort(order.begin(), order.end(), [&](int i, int j) { return sites(i) > sites(j); });
    // a batch of fewer sites is split evenly over the groups that run side by side, unless a group
    // would be too short to be worth a launch of its own
    long long all = 0, in_group = 0, most = kGroupSites;
    for (int i : order) all += sites(i);
    if (all <= kShortSites) most = all;
    else if (all < kChains * kGroupSites) most = (all + kChains - 1) / kChains;
    int total = 0;
    for (int i : order) {
        const lbm::Geom &g = b->geom[i];
        if (b->groups.empty() || in_group + sites(i) > most ||
            b->groups.back().n == lbm::GROUP_LATTICES) {
            b->groups.emplace_back();
            in_group = 0;
        }
        auto &gr = b->groups.back();
        const int tx = (g.nx + lbm::DIRECT_COLS - 1) / lbm::DIRECT_COLS;
        const int tiles = tx * ((g.ny + lbm::STAGED_ROWS - 1) / lbm::STAGED_ROWS);
        gr.lattices.l[gr.n++] = {{buf(b, i, 0), buf(b, i, 1)}, g.nx, g.ny, g.pitch, (unsigned)g.plane, tx, i};
        gr.max_tiles = std::max(gr.max_tiles, tiles);
        in_group += sites(i);
        total += tiles;
    }
    return total;
}

void drop_graphs(lb_batch *b) {
    for (auto &v : b->graphs) {
        for (cudaGraphExec_t g : v)
            if (g) cudaGraphExecDestroy(g);
        v.clear();
    }
}

// room for the graphs of the groups as they are now
void renew_graphs(lb_batch *b) {
    drop_graphs(b);
    b->direct_steps = 0;
    b->no_graphs = false;
    for (auto &v : b->graphs) v.assign((b->groups.size() + kBlockGroups - 1) / kBlockGroups, nullptr);
}

int graph_steps(const lb_batch *b) {
    const size_t n = b->groups.size();
    return n <= 8 ? kGraphSteps : n <= 16 ? kGraphSteps / 2 : kGraphSteps / 4;
}

// A stream beside the batch's, with its priority (launches recorded into a graph keep it).
cudaError_t side_stream(const lb_batch *b, cudaStream_t *st) {
    int priority = 0;
    const cudaError_t e = cudaStreamGetPriority(b->stream, &priority);
    return e != cudaSuccess ? e : cudaStreamCreateWithPriority(st, cudaStreamNonBlocking, priority);
}

// The side streams of several groups.
cudaError_t ensure_side(lb_batch *b) {
    cudaError_t e = cudaSuccess;
    if (!b->fork) e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
    for (int c = 0; c < kChains - 1 && e == cudaSuccess; ++c) {
        if (!b->side[c]) e = side_stream(b, &b->side[c]);
        if (e == cudaSuccess && !b->join[c])
            e = cudaEventCreateWithFlags(&b->join[c], cudaEventDisableTiming);
    }
    return e;
}

// the tensor maps of every lattice's two buffers, for boxes of cols x rows x planes
lb_status make_maps(lb_batch *b, int cols, int rows, int planes, void **d_maps) {
    EncodeTiledFn enc = batch_encode_fn();
    if (!enc) return bfail(b, LB_ECUDA, "cuTensorMapEncodeTiled unavailable");
    std::vector<CUtensorMap> maps(2 * (size_t)b->n);
    const CUtensorMapDataType dt =
        b->prec == LB_FP32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64;
    for (int i = 0; i < b->n; ++i) {
        const lbm::Geom &g = b->geom[i];
        const cuuint64_t dims[3] = {(cuuint64_t)g.pitch, (cuuint64_t)g.ny, 9};
        const cuuint64_t strides[2] = {(cuuint64_t)g.pitch * b->elem, (cuuint64_t)g.plane * b->elem};
        const cuuint32_t box[3] = {(cuuint32_t)cols, (cuuint32_t)rows, (cuuint32_t)planes};
        const cuuint32_t estr[3] = {1, 1, 1};
        for (int w = 0; w < 2; ++w) {
            CUresult r = enc(&maps[2 * i + w], dt, 3, buf(b, i, w), dims, strides, box, estr,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) return bfail(b, LB_ECUDA, "cuTensorMapEncodeTiled failed");
        }
    }
    if (!*d_maps) LB_BCUDA(b, cudaMalloc(d_maps, maps.size() * sizeof(CUtensorMap)));
    LB_BCUDA(b, cudaMemcpy(*d_maps, maps.data(), maps.size() * sizeof(CUtensorMap),
                           cudaMemcpyHostToDevice));
    return LB_OK;
}

void drop_ring(BatchCommon::Ring &r) {
    cudaFree(r.d_items);
    cudaFree(r.d_maps);
    r = {};
}

lb_status make_ring(lb_batch *b, int variant, int rows, BatchCommon::Ring &r) {
    const int tx = lbm::step_variant_tx(variant);
    int occ = 0;
    LB_BCUDA(b, lbm::configure_batch(b->prec, b->eos_kind, variant, &occ));
    std::vector<lbm::BatchItem> items;
    if (!make_items(b, tx, rows, items)) return bfail(b, LB_EINVAL, "bad strip decomposition");
    cudaFree(r.d_items);
    r.d_items = nullptr;
    LB_BCUDA(b, cudaMalloc(&r.d_items, items.size() * sizeof(lbm::BatchItem)));
    LB_BCUDA(b, cudaMemcpy(r.d_items, items.data(), items.size() * sizeof(lbm::BatchItem),
                           cudaMemcpyHostToDevice));
    r.n_items = (int)items.size();
    r.variant = variant;
    r.rows = rows;
    r.grid = std::min(r.n_items, b->num_sms * std::max(occ, 1));
    return make_maps(b, tx + lbm::ghost_of_prec(b->prec) + 4, 1, lbm::step_variant_planes(variant), &r.d_maps);
}

lb_status apply_batch_launch(lb_batch *b, int variant, int rows) {
    if (variant < 0 || variant >= lbm::step_variant_count())
        return bfail(b, LB_EINVAL, "unknown launch variant");
    if (rows <= 0) rows = 16;
    // of the direct kernels batches have the staged tiles, compiled for LB_FP32
    if (variant >= lbm::direct_variant())
        variant = b->prec == LB_FP32 ? lbm::staged_variant() : lbm::default_ring_variant();
    b->few_steps = 0;
    if (variant == lbm::staged_variant()) {
        b->n_items = make_groups(b);
        const lb_status st = make_maps(b, lbm::TILE_BOX_W, lbm::TILE_BOX_ROWS, 3, &b->d_maps);
        if (st != LB_OK) return st;
        b->rows = lbm::STAGED_ROWS;
        b->grid = b->groups.empty() ? 0 : b->groups[0].n * b->groups[0].max_tiles;
        if (b->groups.size() > 1) LB_BCUDA(b, ensure_side(b));
    } else {
        const lb_status st = make_ring(b, variant, rows, b->ring);
        if (st != LB_OK) return st;
        b->n_items = b->ring.n_items;
        b->rows = rows;
        b->grid = b->ring.grid;
        b->groups.assign(b->n_items > 0 ? 1 : 0, {});
    }
    b->variant = variant;
    renew_graphs(b);
    return LB_OK;
}

// the buffer holding lattice i's state: an inactive lattice was set inactive at an even
// step count, so its state stays in buffer 0
int cur(const lb_batch *b, int i) { return b->active[i] ? b->phase : 0; }

template <typename T>
lb_status upload_lattices(lb_batch *b) {
    std::vector<lbm::BatchLattice<T>> t(b->n);
    for (int i = 0; i < b->n; ++i) {
        t[i].g[0] = static_cast<T *>(buf(b, i, 0));
        t[i].g[1] = static_cast<T *>(buf(b, i, 1));
        t[i].P = lbm::to_dev<T>(b->consts[i]);
        t[i].nx = b->geom[i].nx;
        t[i].ny = b->geom[i].ny;
        t[i].pitch = b->geom[i].pitch;
        t[i].plane = (unsigned)b->geom[i].plane;
        t[i].frozen = b->active[i] ? 0 : 1;
    }
    if (!b->d_lats) LB_BCUDA(b, cudaMalloc(&b->d_lats, t.size() * sizeof(t[0])));
    LB_BCUDA(b, cudaMemcpy(b->d_lats, t.data(), t.size() * sizeof(t[0]), cudaMemcpyHostToDevice));
    return LB_OK;
}

void count_steps(lb_batch *b, int n) {
    b->steps += n;
    for (int i = 0; i < b->n; ++i)
        if (b->active[i]) b->lat_steps[i] += n;
}

cudaError_t launch_ring(const lb_batch *b, const BatchCommon::Ring &r, int phase, cudaStream_t st) {
    return lbm::launch_batch_step(b->prec, b->eos_kind, r.variant, r.grid, r.d_maps, b->d_lats, r.d_items,
                                  r.n_items, phase, b->d_errs, st);
}

cudaError_t launch_group(lb_batch *b, const BatchCommon::Group &g, int phase, cudaStream_t st) {
    const cudaError_t e =
        b->variant == lbm::staged_variant()
            ? lbm::batch_tile_f32(b->eos_kind, g.lattices, g.n, g.max_tiles, b->d_maps, b->d_lats, phase,
                                  b->d_errs, st)
            : launch_ring(b, b->ring, phase, st);
    if (e == cudaSuccess) ++b->queued;
    return e;
}

// n steps from phase `phase` of groups first .. last - 1, queued on `main`. Several groups: a group
// takes all its steps before the next one (lattices are independent), so that its state stays in L2,
// and kChains groups run side by side: one computes while another starts a launch or drains one.
cudaError_t queue_groups(lb_batch *b, size_t first, size_t last, int n, int phase, cudaStream_t main) {
    cudaError_t e = cudaSuccess;
    if (last - first <= 1) {
        for (int i = 0; i < n && first < last && e == cudaSuccess; ++i)
            e = launch_group(b, b->groups[first], phase ^ (i & 1), main);
        return e;
    }
    e = cudaEventRecord(b->fork, main);
    for (int c = 0; c < kChains - 1 && e == cudaSuccess; ++c)
        e = cudaStreamWaitEvent(b->side[c], b->fork, 0);
    for (size_t k = first; k < last && e == cudaSuccess; k += kChains)
        for (int i = 0; i < n && e == cudaSuccess; ++i)
            for (size_t c = 0; c < kChains && k + c < last && e == cudaSuccess; ++c)
                e = launch_group(b, b->groups[k + c], phase ^ (i & 1), c == 0 ? main : b->side[c - 1]);
    for (int c = 0; c < kChains - 1; ++c) {       // also after an error: nothing is left unjoined
        cudaError_t j = cudaEventRecord(b->join[c], b->side[c]);
        if (j == cudaSuccess) j = cudaStreamWaitEvent(main, b->join[c], 0);
        if (e == cudaSuccess) e = j;
    }
    return e;
}

// n steps, launched one by one
lb_status launch_steps(lb_batch *b, int n) {
    if (n <= b->few_steps) {
        for (int i = 0; i < n && b->few.n_items > 0; ++i) {
            LB_BCUDA(b, launch_ring(b, b->few, b->phase ^ (i & 1), b->stream));
            ++b->queued;
        }
    } else if (n > 0) {
        LB_BCUDA(b, queue_groups(b, 0, b->groups.size(), n, b->phase, b->stream));
    }
    b->direct_steps = std::min(b->direct_steps + std::min(n, kDirectSteps), kDirectSteps);
    b->phase ^= n & 1;
    count_steps(b, n);
    return LB_OK;
}

// The steps of a block of groups as a graph. The thread may be recording into another stream meanwhile,
// in a mode that forbids it calls that this one makes (and ends the recording at the first): it is
// relaxed for them.
cudaError_t capture_graph(lb_batch *b, size_t first, size_t last, cudaGraphExec_t *exec) {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaError_t e = cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) return e;
    cudaStream_t cap = nullptr;
    cudaGraph_t g = nullptr;
    e = side_stream(b, &cap);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        const long long queued = b->queued;
        e = queue_groups(b, first, last, graph_steps(b), b->phase, cap);
        b->queued = queued;              // recorded only
        const cudaError_t e2 = cudaStreamEndCapture(cap, &g);
        if (e == cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(exec, g, 0);
    if (g) cudaGraphDestroy(g);
    if (cap) cudaStreamDestroy(cap);
    (void)cudaThreadExchangeStreamCaptureMode(&mode);
    return e;
}

// graph_steps steps as graphs, captured when they are first launched: those of a block of groups
// while the GPU takes the steps of the block before. What cannot be captured (no memory for the
// graph) is launched one by one.
lb_status launch_graphs(lb_batch *b) {
    auto &graphs = b->graphs[b->phase];
    for (size_t k = 0; k < graphs.size(); ++k) {
        const size_t first = k * kBlockGroups, last = std::min(first + kBlockGroups, b->groups.size());
        if (!graphs[k] && !b->no_graphs && capture_graph(b, first, last, &graphs[k]) != cudaSuccess) {
            (void)cudaGetLastError();
            graphs[k] = nullptr;
            b->no_graphs = true;
        }
        if (graphs[k]) {
            LB_BCUDA(b, cudaGraphLaunch(graphs[k], b->stream));
            ++b->queued;
        } else {
            LB_BCUDA(b, queue_groups(b, first, last, graph_steps(b), b->phase, b->stream));
        }
    }
    count_steps(b, graph_steps(b));   // even: the phase is unchanged
    return LB_OK;
}

// a capture of the caller's takes the steps launch by launch (a graph launch cannot be captured)
bool capturing(const lb_batch *b) {
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(b->stream, &s) == cudaSuccess) return s != cudaStreamCaptureStatusNone;
    (void)cudaGetLastError();
    return false;
}

lb_status take_steps(lb_batch *b, int n) {
    if (n >= graph_steps(b) && !capturing(b)) {
        if (b->groups.size() > 1 && b->direct_steps < kDirectSteps) {
            const int m = std::min(n, kDirectSteps - b->direct_steps);
            const lb_status s = launch_steps(b, m);
            if (s != LB_OK) return s;
            n -= m;
        }
        for (; n >= graph_steps(b); n -= graph_steps(b)) {
            const lb_status s = launch_graphs(b);
            if (s != LB_OK) return s;
        }
    }
    return launch_steps(b, n);
}

// waits for the stream; h_errs then holds the lattices' error words
lb_status batch_sync(lb_batch *b) {
    LB_BCUDA(b, cudaMemcpyAsync(b->h_errs, b->d_errs, b->n * sizeof(int), cudaMemcpyDeviceToHost,
                                b->stream));
    LB_BCUDA(b, cudaStreamSynchronize(b->stream));
    int any = 0;
    for (int i = 0; i < b->n; ++i) any |= b->h_errs[i];
    if (any & lbm::ERR_TIMEOUT)
        return bfail(b, LB_ETIMEOUT, "a bounded device-side wait gave up", true);
    return LB_OK;   // per-lattice domain errors are reported by lb_batch_errors
}

}  // namespace

extern "C" {

int lb_strip_widths(int nx, int tx, int *widths, int max_strips) {
    if (nx < 1 || tx < 4 || (tx & 3) || !widths) return -1;
    const int ns = (nx + tx - 1) / tx;
    if (ns > max_strips) return -1;
    // m groups of 4 columns (the last one possibly partial) spread as evenly as possible;
    // every strip but the last is a whole number of groups, so all starts are multiples of 4
    const int m = (nx + 3) / 4;
    int used = 0;
    for (int k = 0; k < ns; ++k) {
        const int g = m / ns + (k < m % ns ? 1 : 0);
        widths[k] = 4 * g;
        used += widths[k];
    }
    widths[ns - 1] -= used - nx;   // drop the unused part of the last group
    return ns;
}

lb_status lb_batch_create(lb_batch **out, int n, const lb_lattice_desc *descs, int prec,
                          void *stream) {
    if (!out || n <= 0 || !descs) return LB_EINVAL;
    *out = nullptr;
    if (prec != LB_FP32 && prec != LB_FP64) return LB_EINVAL;
    lb_batch *b = new (std::nothrow) lb_batch();
    if (!b) return LB_ENOMEM;
    b->n = n;
    b->prec = prec;
    b->elem = prec == LB_FP32 ? 4 : 8;
    b->stream = static_cast<cudaStream_t>(stream);
    b->eos_kind = descs[0].eos.kind;
    size_t total = 0;
    for (int i = 0; i < n; ++i) {
        const lb_lattice_desc &d = descs[i];
        if (d.eos.kind != b->eos_kind || d.nx < 3 || d.ny < 3 ||
            9LL * (long long)lb_pitch(d.nx, prec) * d.ny >= (1LL << 32)) {
            delete b;
            return LB_EINVAL;
        }
        if (!(d.kappa >= 0 && d.kappa < 1) || !(d.sigma_force >= 0) ||
            (d.sigma_force != 0 && d.rates.s_zeta != d.rates.s_e)) {
            delete b;
            return LB_EINVAL;
        }
        const double r[6] = {d.rates.s_rho, d.rates.s_e, d.rates.s_zeta, d.rates.s_j,
                             d.rates.s_q, d.rates.s_v};
        for (double s : r)
            if (!(s > 0 && s < 2)) {
                delete b;
                return LB_EINVAL;
            }
        if (d.eos.kind != LB_EOS_EXP && d.G == 0.0) {
            delete b;
            return LB_EINVAL;
        }
        lbm::Geom g;
        g.nx = d.nx;
        g.ny = d.ny;
        g.pitch = (int)lb_pitch(d.nx, prec);
        g.plane = (long long)d.ny * g.pitch;
        g.walls = 0;
        b->geom.push_back(g);
        lbm::Consts c{};
        c.eos_kind = d.eos.kind;
        c.a = d.eos.a;
        c.b4 = d.eos.b / 4.0;
        c.RT = d.eos.R * d.eos.T;
        c.psi0 = d.eos.psi0;
        c.rho0 = d.eos.rho0;
        c.th_v = d.eos.theta_v;
        c.th_m = d.eos.theta_m;
        c.th_l = d.eos.theta_l;
        c.rho1 = d.eos.rho1;
        c.rho2 = d.eos.rho2;
        c.p_rho1 = d.eos.rho1 * d.eos.theta_v;
        c.p_rho2 = c.p_rho1 + (d.eos.rho2 - d.eos.rho1) * d.eos.theta_m;
        c.two_over_G = d.G != 0 ? 2.0 / d.G : 0.0;
        c.G = d.G;
        c.kG2 = d.kappa * d.G / 2.0;
        c.sig_coef = 12.0 * d.sigma_force * d.G * d.G / (1.0 / d.rates.s_e - 0.5);
        c.s_e = d.rates.s_e;
        c.s_z = d.rates.s_zeta;
        c.s_q = d.rates.s_q;
        c.s_v = d.rates.s_v;
        c.stall_row = INT_MIN;
        c.rho_sw = -HUGE_VAL;       // nu(rho) off
        c.s_v_vapour = c.s_v;
        b->consts.push_back(c);
        const size_t bytes = (lb_buffer_bytes(d.nx, d.ny, prec) + 255) / 256 * 256;
        for (int w = 0; w < 2; ++w) {
            b->off[w].push_back(total);
            total += bytes;
        }
        b->stage_sites = std::max(b->stage_sites, (size_t)d.nx * d.ny);
    }
    int dev = 0;
    lb_status s = LB_OK;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&b->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaMalloc(&b->pool, total) != cudaSuccess ||
        cudaMalloc(&b->d_maps, 2 * (size_t)n * sizeof(CUtensorMap)) != cudaSuccess ||
        cudaMalloc(&b->d_errs, n * sizeof(int)) != cudaSuccess ||
        cudaMalloc(&b->d_stage, 3 * b->stage_sites * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&b->d_radius, n * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&b->d_meas, 8 * (size_t)n * sizeof(double)) != cudaSuccess ||
        cudaMallocHost(&b->h_meas, (size_t)n * (9 * sizeof(double) + sizeof(int))) != cudaSuccess ||
        cudaMemset(b->pool, 0, total) != cudaSuccess ||
        cudaMemset(b->d_errs, 0, n * sizeof(int)) != cudaSuccess) {
        lb_batch_free(b);
        return lbm::reported(LB_ENOMEM);
    }
    // one page-locked block: each allocation of one costs about 0.15 ms
    b->h_radius = b->h_meas + 8 * (size_t)n;
    b->h_errs = reinterpret_cast<int *>(b->h_radius + n);
    b->active.assign(n, 1);
    b->lat_steps.assign(n, 0);
    if ((s = make_chunks(b)) != LB_OK) {
        lb_batch_free(b);
        return lbm::reported(s);
    }
    s = prec == LB_FP32 ? upload_lattices<float>(b) : upload_lattices<double>(b);
    if (s == LB_OK) s = apply_batch_launch(b, lbm::staged_variant(), 16);
    if (s != LB_OK) {
        std::fprintf(stderr, "lb_batch_create: %s\n", b->msg.c_str());
        lb_batch_free(b);
        return lbm::reported(s);
    }
    *out = b;
    return LB_OK;
}

lb_status lb_batch_set_launch(lb_batch *b, int variant, int rows) {
    if (!b) return LB_EINVAL;
    if (b->sticky != LB_OK) return b->sticky;
    LB_BCUDA(b, cudaStreamSynchronize(b->stream));
    return apply_batch_launch(b, variant, rows);
}

lb_status lb_batch_get_launch(const lb_batch *b, int *variant, int *rows, int *grid,
                              int *items) {
    if (!b) return LB_EINVAL;
    if (variant) *variant = b->variant;
    if (rows) *rows = b->rows;
    if (grid) *grid = b->grid;
    if (items) *items = b->n_items;
    return LB_OK;
}

lb_status lb_batch_autotune(lb_batch *b, int trial_steps, int *variant, int *rows) {
    if (!b) return LB_EINVAL;
    if (b->sticky != LB_OK) return b->sticky;
    if (trial_steps < 2) trial_steps = 2;
    // the trial launches take real steps of the current states: the pool, the error flags,
    // the phase and the step count are saved first and restored afterwards
    const size_t total = b->off[1].back() +
                         (lb_buffer_bytes(b->geom.back().nx, b->geom.back().ny, b->prec) + 255) / 256 * 256;
    void *saved = nullptr;
    int *saved_errs = nullptr;
    if (cudaMalloc(&saved, total) != cudaSuccess) {
        cudaGetLastError();
        return bfail(b, LB_ENOMEM, "lb_batch_autotune: no device memory for the state copy");
    }
    if (cudaMalloc(&saved_errs, b->n * sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(saved);
        return bfail(b, LB_ENOMEM, "lb_batch_autotune: no device memory for the state copy");
    }
    const int phase0 = b->phase;
    const long long steps0 = b->steps;
    const std::vector<long long> lat_steps0 = b->lat_steps;
    const int v0 = b->variant, r0 = b->rows;
    cudaError_t e = cudaMemcpyAsync(saved, b->pool, total, cudaMemcpyDeviceToDevice, b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(saved_errs, b->d_errs, b->n * sizeof(int), cudaMemcpyDeviceToDevice,
                            b->stream);
    const int cand_rows[] = {8, 12, 16, 24, 32};
    float best = 1e30f, best_ring = 1e30f;   // ms a step
    int bv = v0, br = r0, ring_v = 0, ring_r = 0, few = 0;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    // ms a step of `calls` calls of `steps` steps, 0 if they cannot be launched
    auto timed = [&](int calls, int steps) {
        float ms = 0;
        if (launch_steps(b, steps) != LB_OK) return 0.f;           // warm-up
        cudaEventRecord(e0, b->stream);
        for (int i = 0; i < calls; ++i)
            if (launch_steps(b, steps) != LB_OK) return 0.f;
        cudaEventRecord(e1, b->stream);
        e = cudaEventSynchronize(e1);
        if (e == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
        return ms / (float)(calls * steps);
    };
    for (int v = 0; v < lbm::step_variant_count() && e == cudaSuccess; ++v) {
        for (int r : cand_rows) {
            if (v == lbm::direct_variant()) break;   // batches take the staged tiles
            if (v == lbm::staged_variant() && (b->prec != LB_FP32 || r != cand_rows[0])) break;
            if (apply_batch_launch(b, v, r) != LB_OK) continue;
            // the groups of the staged tiles keep their state in L2 over the steps of a call: they
            // are timed over a call of some length
            const float ms = v == lbm::staged_variant() ? timed(1, std::max(trial_steps, 16)) : timed(trial_steps, 1);
            if (ms > 0 && ms < best) {
                best = ms;
                bv = v;
                br = b->rows;
            }
            if (ms > 0 && ms < best_ring && v < lbm::direct_variant()) {
                best_ring = ms;
                ring_v = v;
                ring_r = r;
            }
        }
    }
    // In calls of one step or a few nothing stays in L2, and the groups' many launches take longer than
    // the ring kernel's one where memory is the bound: staged / ring, us a step, 512 lattices of 64^2 to
    // 512^2 812 / 741 (calls of four 658), 2 of 1024^2 36.2 / 29.3 (29.8), 60 of 64^2 to 512^2 97.9 / 78.7
    // (73.5); 24 of 128^2 11.2 / 12.9.
    if (bv == lbm::staged_variant() && best_ring < 1e30f && e == cudaSuccess &&
        apply_batch_launch(b, bv, br) == LB_OK && b->groups.size() > 1)
        for (int k = 1; k <= 4 && e == cudaSuccess && best_ring < timed(8 / k, k); k *= 2) few = k;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    // put the states back (whatever the trials did)
    cudaError_t e2 = cudaMemcpyAsync(b->pool, saved, total, cudaMemcpyDeviceToDevice, b->stream);
    if (e2 == cudaSuccess)
        e2 = cudaMemcpyAsync(b->d_errs, saved_errs, b->n * sizeof(int), cudaMemcpyDeviceToDevice,
                             b->stream);
    if (e2 == cudaSuccess) e2 = cudaStreamSynchronize(b->stream);
    cudaFree(saved);
    cudaFree(saved_errs);
    b->phase = phase0;
    b->steps = steps0;
    b->lat_steps = lat_steps0;
    if (e != cudaSuccess) return bfail(b, LB_ECUDA, cudaGetErrorString(e));
    if (e2 != cudaSuccess) return bfail(b, LB_ECUDA, cudaGetErrorString(e2));
    lb_status s = apply_batch_launch(b, bv, br);
    if (s == LB_OK && few > 0) s = make_ring(b, ring_v, ring_r, b->few);
    if (s != LB_OK) return s;
    b->few_steps = few;
    if (variant) *variant = bv;
    if (rows) *rows = br;
    return LB_OK;
}

lb_status lb_batch_set_rho_u(lb_batch *b, int i, const double *rho, const double *ux,
                             const double *uy) {
    if (!b || i < 0 || i >= b->n || !rho || !ux || !uy) return LB_EINVAL;
    if (b->sticky != LB_OK) return b->sticky;
    const lbm::Geom &g = b->geom[i];
    const size_t n = (size_t)g.nx * g.ny;
    LB_BCUDA(b, cudaMemcpyAsync(b->d_stage, rho, n * sizeof(double), cudaMemcpyHostToDevice, b->stream));
    LB_BCUDA(b, cudaMemcpyAsync(b->d_stage + n, ux, n * sizeof(double), cudaMemcpyHostToDevice, b->stream));
    LB_BCUDA(b, cudaMemcpyAsync(b->d_stage + 2 * n, uy, n * sizeof(double), cudaMemcpyHostToDevice, b->stream));
    // the per-lattice error word doubles as the init kernel's domain flag
    LB_BCUDA(b, lbm::launch_init_feq(b->prec, b->consts[i], g, b->d_stage, b->d_stage + n,
                                     b->d_stage + 2 * n, buf(b, i, cur(b, i) ^ 1), b->d_errs + i,
                                     b->stream));
    LB_BCUDA(b, lbm::launch_unstream(b->prec, g, buf(b, i, cur(b, i) ^ 1), buf(b, i, cur(b, i)),
                                     false, b->stream));
    LB_BCUDA(b, cudaStreamSynchronize(b->stream));
    int e = 0;
    LB_BCUDA(b, cudaMemcpy(&e, b->d_errs + i, sizeof(int), cudaMemcpyDeviceToHost));
    if (e & lbm::ERR_DOMAIN) return bfail(b, LB_EDOMAIN, "lattice density outside the EOS branch");
    return LB_OK;
}

lb_status lb_batch_step(lb_batch *b, int n) {
    const lbm::NvtxRange nvtx_range("lb_batch_step");
    if (!b || n < 0) return LB_EINVAL;
    if (b->sticky != LB_OK) return b->sticky;
    const long long queued = b->queued;
    const lb_status s = take_steps(b, n);
    // some lattices have gone on and others not: nothing can be made of the batch any more
    if (s != LB_OK && b->queued != queued) b->sticky = s;
    return s;
}

lb_status lb_batch_sync(lb_batch *b) {
    if (!b) return LB_EINVAL;
    if (b->sticky != LB_OK) return b->sticky;
    return batch_sync(b);
}

lb_status lb_batch_errors(lb_batch *b, int *flags) {
    if (!b || !flags) return LB_EINVAL;
    lb_status s = batch_sync(b);
    if (s != LB_OK && s != LB_ETIMEOUT) return s;
    std::memcpy(flags, b->h_errs, b->n * sizeof(int));
    return s;
}

lb_status lb_batch_get_rho(lb_batch *b, int i, double *rho) {
    if (!b || i < 0 || i >= b->n || !rho) return LB_EINVAL;
    if (b->sticky != LB_OK) return b->sticky;
    const lbm::Geom &g = b->geom[i];
    const size_t n = (size_t)g.nx * g.ny;
    LB_BCUDA(b, lbm::launch_macro_fields(b->prec, b->consts[i], g, buf(b, i, cur(b, i)), nullptr,
                                         b->d_stage, nullptr, nullptr, b->stream));
    LB_BCUDA(b, cudaMemcpyAsync(rho, b->d_stage, n * sizeof(double), cudaMemcpyDeviceToHost, b->stream));
    return batch_sync(b);
}

lb_status lb_batch_get_populations(lb_batch *b, int i, void *dst, size_t bytes) {
    if (!b || i < 0 || i >= b->n || !dst) return LB_EINVAL;
    if (b->sticky != LB_OK) return b->sticky;
    const lbm::Geom &g = b->geom[i];
    const size_t row = (size_t)g.nx * b->elem;
    if (bytes != 9 * (size_t)g.ny * row) return bfail(b, LB_EINVAL, "size mismatch");
    // the spare buffer of lattice i receives the pulled populations in the host layout
    // (free between steps), then one contiguous copy
    void *spare = buf(b, i, cur(b, i) ^ 1);
    LB_BCUDA(b, lbm::launch_stream(b->prec, g, buf(b, i, cur(b, i)), spare, true, b->stream));
    LB_BCUDA(b, cudaMemcpyAsync(dst, spare, bytes, cudaMemcpyDeviceToHost, b->stream));
    return batch_sync(b);
}

lb_status lb_batch_measure(lb_batch *b, const double *radius, double *out) {
    const lbm::NvtxRange nvtx_range("lb_batch_measure");
    if (!b || !radius || !out) return LB_EINVAL;
    if (b->sticky != LB_OK) return b->sticky;
    // every call that uses h_radius waits for its stream before it returns
    std::memcpy(b->h_radius, radius, b->n * sizeof(double));
    LB_BCUDA(b, cudaMemcpyAsync(b->d_radius, b->h_radius, b->n * sizeof(double),
                                cudaMemcpyHostToDevice, b->stream));
    LB_BCUDA(b, lbm::launch_batch_measure(b->prec, b->eos_kind, b->d_lats, b->n, b->d_chunks,
                                          b->d_first, b->n_chunks, b->phase, b->d_radius,
                                          b->d_partials, b->d_meas, b->stream));
    LB_BCUDA(b, cudaMemcpyAsync(b->h_meas, b->d_meas, 8 * (size_t)b->n * sizeof(double),
                                cudaMemcpyDeviceToHost, b->stream));
    lb_status s = batch_sync(b);
    if (s != LB_OK) return s;
    for (int i = 0; i < b->n; ++i)
        lbm::droplet_results(b->h_meas + 8 * (size_t)i, (double)b->geom[i].nx * b->geom[i].ny,
                             b->h_errs[i] != 0, out + 8 * (size_t)i);
    return LB_OK;
}

lb_status lb_batch_set_active(lb_batch *b, const unsigned char *active) {
    if (!b || !active) return LB_EINVAL;
    if (b->sticky != LB_OK) return b->sticky;
    if (b->steps & 1)
        return bfail(b, LB_EINVAL, "lb_batch_set_active: call at an even step count");
    LB_BCUDA(b, cudaStreamSynchronize(b->stream));   // no queued step reads the old items
    for (int i = 0; i < b->n; ++i) b->active[i] = active[i] ? 1 : 0;
    lb_status s = b->prec == LB_FP32 ? upload_lattices<float>(b) : upload_lattices<double>(b);
    if (s != LB_OK) return s;
    const int few = b->few_steps;
    if ((s = apply_batch_launch(b, b->variant, b->rows)) != LB_OK || few == 0) return s;
    if ((s = make_ring(b, b->few.variant, b->few.rows, b->few)) == LB_OK) b->few_steps = few;
    return s;
}

long long lb_batch_lattice_steps(const lb_batch *b, int i) {
    return (b && i >= 0 && i < b->n) ? b->lat_steps[i] : -1;
}

long long lb_batch_steps_done(const lb_batch *b) { return b ? b->steps : 0; }

int lb_batch_size(const lb_batch *b) { return b ? b->n : 0; }

const char *lb_batch_last_error(const lb_batch *b) { return b ? b->msg.c_str() : "no batch"; }

void lb_batch_free(lb_batch *b) {
    if (!b) return;
    if (b->stream) cudaStreamSynchronize(b->stream);
    else cudaDeviceSynchronize();
    drop_graphs(b);
    for (int c = 0; c < kChains - 1; ++c) {
        if (b->side[c]) cudaStreamDestroy(b->side[c]);
        if (b->join[c]) cudaEventDestroy(b->join[c]);
    }
    if (b->fork) cudaEventDestroy(b->fork);
    cudaFree(b->pool);
    cudaFree(b->d_maps);
    cudaFree(b->d_lats);
    drop_ring(b->ring);
    drop_ring(b->few);
    cudaFree(b->d_errs);
    cudaFree(b->d_stage);
    cudaFree(b->d_radius);
    cudaFree(b->d_meas);
    cudaFree(b->d_chunks);
    cudaFreeHost(b->h_meas);
    cudaFree(b->d_first);
    cudaFree(b->d_partials);
    delete b;
}

}  // extern "C"
