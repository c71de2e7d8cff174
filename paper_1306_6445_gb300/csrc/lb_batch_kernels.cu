// Batched-lattice kernels: the persistent step over work items with the whole-row ring
// (FP32, FP64; the stage ring is in lb_batch_stage.cu) and the per-lattice Laplace
// measurement.
#include "lb_step.cuh"

namespace lbm {

namespace {

// Laplace sums of a chunk of rows of one lattice (fixed per-thread order and fixed tree, so
// deterministic). Inside: r < R/2; outside: r > R + 0.3 min(nx,ny)/2; p = rho/3 + (G/2) psi^2,
// summed as sums of rho and psi^2.
// What bounds it: memory (36 bytes a site in FP32) next to the FP64 pipe (2 operations per
// clock and SM): 4 FP64 operations a site are left (two conversions, two sums). One CTA per
// lattice with a root and a division per site took 8.97 ms for 512 lattices of 64^2 to 512^2
// (51.6 M sites); in chunks of 8192 sites 64 steps and a measurement take 49.9 against 57.8 ms.
template <typename T, int EOS>
__global__ void __launch_bounds__(RED_THREADS)
k_batch_measure(const BatchLattice<T> *__restrict__ lats, const MeasureChunk *__restrict__ chunks,
                int phase, const double *__restrict__ radius, double *__restrict__ partials) {
    __shared__ long long limit[2];
    const MeasureChunk ch = chunks[blockIdx.x];
    const BatchLattice<T> &L = lats[ch.lat];
    const DevConsts<T> P = L.P;
    const int nx = L.nx, ny = L.ny, pitch = L.pitch;
    const T *__restrict__ g = L.g[L.frozen ? 0 : phase];
    if (threadIdx.x < 2) {
        const double R = radius[ch.lat];
        limit[threadIdx.x] = threadIdx.x == 0 ? quarters_below(0.5 * R) : quarters_above(R + 0.3 * 0.5 * min(nx, ny));
    }
    __syncthreads();
    const long long d_in = limit[0], d_out = limit[1];
    double m_in = 0, m_out = 0, m_rest = 0, q_in = 0, q_out = 0;
    int n_in = 0, n_out = 0, n_bad = 0;
    const unsigned n = (unsigned)ch.rows * (unsigned)nx;
    for (unsigned i = threadIdx.x; i < n; i += RED_THREADS) {
        const unsigned row = i / (unsigned)nx;
        const int x = (int)(i - row * (unsigned)nx), y = ch.row0 + (int)row;
        T v[9];
#pragma unroll
        for (int a = 0; a < 9; ++a) v[a] = pull_padded<T, 0>(g, a, x, y, ny, pitch, L.plane);
        const T rho = sum9(v);
        bool bad = false;
        const T psi = eos_psi<T, EOS>(rho, P, bad);
        const double dr = double(rho), ds = double(psi);
        const int a = 2 * x - (nx - 1), b = 2 * y - (ny - 1);
        const long long d = (long long)a * a + (long long)b * b;
        if (d < d_in) {
            m_in += dr;
            q_in = fma(ds, ds, q_in);
            ++n_in;
        } else if (d >= d_out) {
            m_out += dr;
            q_out = fma(ds, ds, q_out);
            ++n_out;
        } else {
            m_rest += dr;
        }
        if (bad || !(rho == rho) || !(psi == psi)) ++n_bad;
    }
    droplet_combine(m_in, m_out, m_rest, q_in, q_out, n_in, n_out, n_bad, double(P.G),
                    partials + (size_t)blockIdx.x * 8);
}

// Sum of the chunks of each lattice in a fixed order: warp k of CTA i adds quantity k.
__global__ void __launch_bounds__(RED_THREADS)
k_batch_measure_sum(const double *__restrict__ partials, const int *__restrict__ first,
                    double *__restrict__ out) {
    static_assert(RED_THREADS == 8 * 32, "one warp per quantity");
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c0 = first[blockIdx.x], c1 = first[blockIdx.x + 1];
    double t = 0;
    for (int c = c0 + lane; c < c1; c += 32) t += partials[(size_t)c * 8 + k];
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) t += __shfl_xor_sync(0xffffffffu, t, w);
    if (lane == 0) out[blockIdx.x * 8 + k] = t;
}

}  // namespace

cudaError_t launch_batch_measure(int prec, int eos_kind, const void *lats, int n_lat,
                                 const MeasureChunk *chunks, const int *first, int n_chunks,
                                 int phase, const double *radius, double *partials, double *out,
                                 cudaStream_t st) {
#define LB_BM(T, EOSK)                                                                         \
    k_batch_measure<T, EOSK><<<n_chunks, RED_THREADS, 0, st>>>(                                \
        static_cast<const BatchLattice<T> *>(lats), chunks, phase, radius, partials)
    if (prec == LB_FP32) {
        if (eos_kind == LB_EOS_CS) LB_BM(float, LB_EOS_CS);
        else if (eos_kind == LB_EOS_EXP) LB_BM(float, LB_EOS_EXP);
        else LB_BM(float, LB_EOS_PIECEWISE);
    } else {
        if (eos_kind == LB_EOS_CS) LB_BM(double, LB_EOS_CS);
        else if (eos_kind == LB_EOS_EXP) LB_BM(double, LB_EOS_EXP);
        else LB_BM(double, LB_EOS_PIECEWISE);
    }
#undef LB_BM
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_batch_measure_sum<<<n_lat, RED_THREADS, 0, st>>>(partials, first, out);
    return cudaGetLastError();
}


LB_BATCH_UNIT(f32, float, 0)
LB_BATCH_UNIT(f64, double, 0)

}  // namespace lbm
