// Many time steps of a small FP32 lattice in one launch: the lattice lives in the shared memory of
// one thread-block cluster (k_cluster_steps). Same arithmetic and results, bit for bit, as the step
// kernels of lb_step.cuh and lb_tile.cuh.
#include "lb_step.cuh"

namespace lbm {

namespace {

constexpr int CL_SIZE = 16;           // CTAs of the cluster
constexpr int CL_MAX_THREADS = 512;   // of a CTA: as many as it has site pairs, in warps
constexpr int CL_SMEM_MOST = 200 * 1024;

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// wait until every thread of the cluster is here; what each wrote before (to its own CTA's shared
// memory or another's) is visible to all afterwards
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// address of the same shared-memory variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t remote_addr(const void *p, unsigned rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void store_remote(uint32_t addr, V2<float> v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.lo()), "f"(v.hi()) : "memory");
}

// n_steps time steps of one lattice (periodic in x, even nx; BC 0 or 1): CTA c of the cluster owns
// rows ny c / 16 .. ny (c + 1) / 16 - 1. Shared memory: the nine stored planes of its rows with one
// halo row on either side ([9][rows + 2][nx]; only the plane group pulled across is kept current
// there), and psi of the same rows. A step: pull the thread's pairs (kept in registers) and form
// psi, edge rows also into the neighbours' halo; cluster barrier; collide and store in place, edge
// rows also into the neighbours' halo; cluster barrier.
// What bounds it: two cluster barriers and the chain between them: 1.1 us a step for 64^2, 1.9 for
// 128^2, where a launch per step takes 2.3. A thread has one pair, a CTA at most 512 (16 384 sites
// in all): with two pairs per thread 140^2 took 2.3, 160^2 2.6 us, no less than the launches.
template <int EOS, int BC>
__global__ void __launch_bounds__(CL_MAX_THREADS, 1)
k_cluster_steps(const float *gin, float *gout,          // (may be the same)
                const __grid_constant__ DevConsts<float> P, const int nx, const int ny,
                const int pitch, const unsigned plane, const int n_steps, int *__restrict__ err) {
    extern __shared__ __align__(16) float cl_smem[];
    using T = float;
    const unsigned rank = cluster_rank();
    const int y0 = (int)(ny * rank / CL_SIZE), rows = (int)(ny * (rank + 1) / CL_SIZE) - y0;
    const int max_rows = (ny + CL_SIZE - 1) / CL_SIZE;       // the same layout in every CTA
    const int RS = nx, PS = (max_rows + 2) * nx;              // row and plane stride
    float *g = cl_smem, *ps = cl_smem + 9 * PS;               // row r of the CTA: r + 1
    const unsigned below = rank == 0 ? CL_SIZE - 1 : rank - 1, above = rank + 1 == CL_SIZE ? 0 : rank + 1;
    const int rows_below = (int)(ny * (below + 1) / CL_SIZE) - (int)(ny * below / CL_SIZE);
    const bool has_below = BC == 0 || rank > 0, has_above = BC == 0 || rank + 1 < CL_SIZE;
    // my first row is the row above the last of `below`; my last row lies below the first of `above`
    const uint32_t g_below = remote_addr(g, below) + 4u * (unsigned)((rows_below + 1) * RS);
    const uint32_t g_above = remote_addr(g, above);
    const uint32_t ps_below = remote_addr(ps, below) + 4u * (unsigned)((rows_below + 1) * RS);
    const uint32_t ps_above = remote_addr(ps, above);

    // the thread's pair: row r of the CTA, columns x, x + 1, and their neighbours x - 1, x + 2
    const bool act = (int)threadIdx.x < rows * (nx / 2);
    const int r = act ? (int)threadIdx.x / (nx / 2) : 0, x = act ? 2 * ((int)threadIdx.x - r * (nx / 2)) : 0;
    const int xl = x == 0 ? nx - 1 : x - 1, xr = x + 2 == nx ? 0 : x + 2, y = y0 + r;

    // the state: own rows and the halo rows (rows beyond a wall are not read)
    for (int i = (int)threadIdx.x; i < 9 * (rows + 2) * (nx / 2); i += (int)blockDim.x) {
        const int p = i / ((rows + 2) * (nx / 2)), q = i - p * ((rows + 2) * (nx / 2));
        const int r = q / (nx / 2), x = 2 * (q - r * (nx / 2));
        int y = y0 + r - 1;
        if (BC == 0) y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        if (y >= 0 && y < ny)
            *reinterpret_cast<float2 *>(g + p * PS + r * RS + x) = *reinterpret_cast<const float2 *>(
                gin + (size_t)p * plane + (unsigned)y * (unsigned)pitch + (unsigned)(x + GH<T>));
    }
    cluster_sync();

    bool bad = false;
    V2<T> f[9];
    auto at = [&](int a, int dr) { return g + plane_of(a) * PS + (r + 1 + dr) * RS; };
#pragma unroll 1
    for (int step = 0; step < n_steps; ++step) {
        if (act) {
            auto mid = [&](int a, int dr) { return lds_pair<T>(at(a, dr) + x); };
            auto lft = [&](int a, int dr) { const T *p = at(a, dr); return V2<T>(p[xl], p[x]); };
            auto rgt = [&](int a, int dr) { const T *p = at(a, dr); return V2<T>(p[x + 1], p[xr]); };
            f[0] = mid(0, 0);
            f[1] = lft(1, 0);
            f[3] = rgt(3, 0);
            if (BC == 1 && y == 0) {
                f[2] = mid(4, 0);
                f[5] = mid(7, 0);
                f[6] = mid(8, 0);
            } else {
                f[2] = mid(2, -1);
                f[5] = lft(5, -1);
                f[6] = rgt(6, -1);
            }
            if (BC == 1 && y == ny - 1) {
                f[4] = mid(2, 0);
                f[7] = mid(5, 0);
                f[8] = mid(6, 0);
            } else {
                f[4] = mid(4, 1);
                f[7] = rgt(7, 1);
                f[8] = lft(8, 1);
            }
            const V2<T> psi = eos_psi2<T, EOS>(rho_pair(f), P, true, bad);
            store_pair<T>(ps + (r + 1) * RS + x, psi, true);
            if (r == 0 && has_below) store_remote(ps_below + 4u * (unsigned)x, psi);
            if (r == rows - 1 && has_above) store_remote(ps_above + 4u * (unsigned)x, psi);
        }
        cluster_sync();               // psi is complete, every population has been pulled
        if (act) {
            const T *p0 = ps + (r + 1) * RS;
            const T *pm = BC == 1 && y == 0 ? p0 : p0 - RS;
            const T *pp = BC == 1 && y == ny - 1 ? p0 : p0 + RS;
            const V2<T> m0 = lds_pair<T>(pm + x), z0 = lds_pair<T>(p0 + x), q0 = lds_pair<T>(pp + x);
            V2<T> pn[9];
            pn[0] = z0;
            pn[1] = V2<T>(z0.hi(), p0[xr]);
            pn[2] = q0;
            pn[3] = V2<T>(p0[xl], z0.lo());
            pn[4] = m0;
            pn[5] = V2<T>(q0.hi(), pp[xr]);
            pn[6] = V2<T>(pp[xl], q0.lo());
            pn[7] = V2<T>(pm[xl], m0.lo());
            pn[8] = V2<T>(m0.hi(), pm[xr]);
            collide<T>(f, pn, P);
#pragma unroll
            for (int a = 0; a < 9; ++a) store_pair<T>(const_cast<T *>(at(a, 0)) + x, f[a], true);
            if (r == 0 && has_below) {            // the row below pulls planes 4, 7, 8 from here
#pragma unroll
                for (int a = 0; a < 9; ++a)
                    if (EYv(a) < 0) store_remote(g_below + 4u * (unsigned)(plane_of(a) * PS + x), f[a]);
            }
            if (r == rows - 1 && has_above) {     // the row above pulls planes 2, 5, 6 from here
#pragma unroll
                for (int a = 0; a < 9; ++a)
                    if (EYv(a) > 0) store_remote(g_above + 4u * (unsigned)(plane_of(a) * PS + x), f[a]);
            }
        }
        cluster_sync();               // the new state is complete; nothing is in flight after the last step
    }

    // back to memory (f holds what was stored last), with the images of the edge columns
    if (act) {
        const unsigned rowi = (unsigned)y * (unsigned)pitch;
#pragma unroll
        for (int a = 0; a < 9; ++a)
            store_pair<T>(gout + (size_t)plane_of(a) * plane + rowi + (unsigned)(x + GH<T>), f[a], true);
        store_ghosts<T, BC, false>(gout, f, x, rowi, nx, plane, true, 0u);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, ERR_DOMAIN);
}

int cluster_smem(const Geom &g) { return 10 * ((g.ny + CL_SIZE - 1) / CL_SIZE + 2) * g.nx * (int)sizeof(float); }

int cluster_pairs(const Geom &g) { return (g.ny + CL_SIZE - 1) / CL_SIZE * (g.nx / 2); }   // most of one CTA

template <int EOS, int BC>
cudaError_t cluster_launch(const Consts &c, const Geom &g, const void *gin, void *gout, int n_steps,
                           int *err, cudaStream_t st, bool probe) {
    auto kern = k_cluster_steps<EOS, BC>;
    const int smem = cluster_smem(g);
    // the kernel's limit, not this lattice's size: contexts of several threads share the attribute
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, CL_SMEM_MOST);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL_SIZE);
    cfg.blockDim = dim3((cluster_pairs(g) + 31) / 32 * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL_SIZE;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (probe) {
        int n = 0;
        e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
        return e != cudaSuccess ? e : n > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
    }
    return cudaLaunchKernelEx(&cfg, kern, static_cast<const float *>(gin), static_cast<float *>(gout),
                              to_dev<float>(c), g.nx, g.ny, g.pitch, (unsigned)g.plane, n_steps, err);
}

template <int EOS>
cudaError_t cluster_bc(const Consts &c, const Geom &g, const void *gin, void *gout, int n_steps,
                       int *err, cudaStream_t st, bool probe) {
    return g.walls == 0 ? cluster_launch<EOS, 0>(c, g, gin, gout, n_steps, err, st, probe)
                        : cluster_launch<EOS, 1>(c, g, gin, gout, n_steps, err, st, probe);
}

cudaError_t cluster_dispatch(const Consts &c, const Geom &g, const void *gin, void *gout, int n_steps,
                             int *err, cudaStream_t st, bool probe) {
    switch (c.eos_kind) {
        case LB_EOS_CS: return cluster_bc<LB_EOS_CS>(c, g, gin, gout, n_steps, err, st, probe);
        case LB_EOS_EXP: return cluster_bc<LB_EOS_EXP>(c, g, gin, gout, n_steps, err, st, probe);
        default: return cluster_bc<LB_EOS_PIECEWISE>(c, g, gin, gout, n_steps, err, st, probe);
    }
}

}  // namespace

// Periodic lattices and walls in FP32, of even width (pairs do not straddle the seam), with a row
// for every CTA and no more pairs than it has threads.
bool cluster_fits(int prec, const Consts &c, const Geom &g) {
    if (prec != LB_FP32 || g.walls == 2 || (g.nx & 1) || g.nx < 4 || g.ny < CL_SIZE) return false;
    if ((long long)g.nx * g.ny > CL_SIZE * 2ll * CL_MAX_THREADS) return false;
    if (cluster_pairs(g) > CL_MAX_THREADS || cluster_smem(g) > CL_SMEM_MOST) return false;
    if (cluster_dispatch(c, g, nullptr, nullptr, 0, nullptr, nullptr, true) == cudaSuccess) return true;
    (void)cudaGetLastError();
    return false;
}

cudaError_t launch_cluster_steps(const Consts &c, const Geom &g, const void *gin, void *gout,
                                 int n_steps, int *err, cudaStream_t st) {
    return cluster_dispatch(c, g, gin, gout, n_steps, err, st, false);
}

}  // namespace lbm
