// Surrogate network (lb_mlp_*): 3 -> 64 -> 64 -> 3 GELU MLP mapping (T/T_c, kappa, tau_v)
// to (sigma, rho_l, rho_v), trained on the GPU by hand-written kernels:
//   k_mlp_prepare  one CTA: FP64 means / scales of the input features
//                  (ln(1 - T/T_c), ln(1 - kappa), tau_v) and of the transformed targets,
//                  standardised copies (float)
//   k_mlp_grad     forward + backward over tiles of 16 samples, one CTA or a cluster of four
//                  each, which sums the tile's gradient and writes one partial vector
//   k_mlp_adam     sums the partials in a fixed order, Adam update of the FP32 master
//                  copy, refreshes the BF16 image used by the next forward pass
//   k_mlp_forward  inference, one warp per sample or pair of samples
//   k_mlp_invert   bisection on kappa for a target sigma, one warp per query or pair
// The weights are read as BF16 and every product is accumulated in FP32 (fmaf; in the order of
// the sums' indices, the output layer of inference over a fixed butterfly of the lanes).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "lb_internal.h"
#include "lb_mlp.h"

namespace {

constexpr int IN = LB_MLP_IN, H = LB_MLP_HIDDEN, OUT = LB_MLP_OUT, NP = LB_MLP_PARAMS;
constexpr int OW1 = 0, OB1 = OW1 + H * IN, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H,
              OB3 = OW3 + OUT * H;
static_assert(OB3 + OUT == NP, "parameter layout");

constexpr int kTile = 16;          // samples per tile of k_mlp_grad
constexpr int kSplit = 4;          // CTAs that share a tile while the grid leaves room (a cluster)
constexpr int kThreads = 256;      // k_mlp_grad block
constexpr int kMaxGradCtas = 304;  // 2 x 152 SMs: bounds the partial-gradient buffer
constexpr int kW2Pitch = H + 4;    // padded rows of W2 in shared memory (16-byte rows, no bank conflicts)
constexpr int kGraphSteps = 50;
constexpr int kMaxSamples = 1 << 20;
constexpr int kMaxForward = 1 << 22;
constexpr int kBisect = 40;

struct MlpNorm {
    float in_mean[3], in_scale[3], out_mean[3], out_scale[3];
};

struct MlpState {
    int step;          // Adam step count (incremented by the first CTA of k_mlp_grad)
    int n;             // resident samples
    float lr, beta1, beta2, eps;
    float loss;        // loss of the last forward pass of k_mlp_grad (set by k_mlp_adam)
    int pad;
    double pow1, pow2; // beta1^step, beta2^step of this step (advanced with step)
};

__device__ __forceinline__ float gelu(float z) {
    return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f));
}

// d/dz [z Phi(z)] = Phi(z) + z phi(z)
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f))
           + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// Weights as float in shared memory; W2 rows padded to kW2Pitch.
struct SmemW {
    __align__(16) float w2[H * kW2Pitch];
    float w1[H * IN], b1[H], b2[H], w3[OUT * H], b3[4];
};

__device__ __forceinline__ void load_weights(SmemW &w, const __nv_bfloat16 *__restrict__ wbf) {
    static_assert(OW2 * 2 % 16 == 0 && H % 8 == 0, "W2 is read in 16-byte words of one row");
    const uint4 *w2 = reinterpret_cast<const uint4 *>(wbf + OW2);
#pragma unroll
    for (int p = threadIdx.x; p < H * H / 8; p += kThreads) {
        const uint4 u = w2[p];
        const unsigned v[4] = {u.x, u.y, u.z, u.w};
        float4 *d = reinterpret_cast<float4 *>(&w.w2[(p / (H / 8)) * kW2Pitch + (p % (H / 8)) * 8]);
#pragma unroll
        for (int e = 0; e < 2; ++e)
            d[e] = make_float4(__uint_as_float(v[2 * e] << 16), __uint_as_float(v[2 * e] & 0xffff0000u),
                               __uint_as_float(v[2 * e + 1] << 16),
                               __uint_as_float(v[2 * e + 1] & 0xffff0000u));
    }
    for (int p = threadIdx.x; p < OW2; p += kThreads) {
        const float v = __bfloat162float(wbf[p]);
        if (p < OB1) w.w1[p] = v;
        else w.b1[p - OB1] = v;
    }
    for (int p = OB2 + threadIdx.x; p < NP; p += kThreads) {
        const float v = __bfloat162float(wbf[p]);
        if (p < OW3) w.b2[p - OB2] = v;
        else if (p < OB3) w.w3[p - OW3] = v;
        else w.b3[p - OB3] = v;
    }
}

// output c of one sample from the lanes' second-layer activations (the same in every lane)
__device__ __forceinline__ float output_unit(float2 w3, float b3, float2 g) {
    float p = fmaf(w3.y, g.y, w3.x * g.x);
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) p += __shfl_xor_sync(0xffffffffu, p, m);
    return p + b3;
}

// Input features (ln(1 - T/T_c), ln(1 - kappa), tau_v) in float, as inference computes them.
__device__ __forceinline__ float input_feature(float v, int c) {
    return c == 2 ? v : log1pf(-v);
}

// ---------------------------------------------------------------------------------
// Data preparation: one CTA of 512 threads. Two-pass FP64 mean / variance with a fixed
// reduction tree, the scale rule of the header, then standardised float copies in place.
// ---------------------------------------------------------------------------------
constexpr int kPrepThreads = 512;

__device__ void block_sum6(double (&v)[6], double (*red)[6]) {
    const int t = threadIdx.x;
    for (int c = 0; c < 6; ++c) red[t][c] = v[c];
    __syncthreads();
    for (int s = kPrepThreads / 2; s > 0; s >>= 1) {
        if (t < s)
            for (int c = 0; c < 6; ++c) red[t][c] += red[t + s][c];
        __syncthreads();
    }
    for (int c = 0; c < 6; ++c) v[c] = red[0][c];
    __syncthreads();
}

__global__ void __launch_bounds__(kPrepThreads)
k_mlp_prepare(float *__restrict__ x, float *__restrict__ y, int n, MlpNorm *__restrict__ norm) {
    __shared__ double red[kPrepThreads][6];
    const int t = threadIdx.x;
    double acc[6] = {0, 0, 0, 0, 0, 0};
    auto feature = [&](int i, int c) -> double {
        const double v = (double)x[3 * i + c];
        return c == 2 ? v : log1p(-v);
    };
    auto target = [&](int i, int c) -> double {
        const double v = (double)y[3 * i + c];
        return c == 1 ? v : log(v);
    };
    for (int i = t; i < n; i += kPrepThreads)
        for (int c = 0; c < 3; ++c) {
            acc[c] += feature(i, c);
            acc[3 + c] += target(i, c);
        }
    block_sum6(acc, red);
    double mean[6];
    for (int c = 0; c < 6; ++c) mean[c] = acc[c] / n;
    double sq[6] = {0, 0, 0, 0, 0, 0};
    for (int i = t; i < n; i += kPrepThreads)
        for (int c = 0; c < 3; ++c) {
            const double dx = feature(i, c) - mean[c];
            const double dt = target(i, c) - mean[3 + c];
            sq[c] += dx * dx;
            sq[3 + c] += dt * dt;
        }
    block_sum6(sq, red);
    __shared__ float nm[12];
    if (t == 0) {
        for (int c = 0; c < 6; ++c) {
            const double s = sqrt(sq[c] / n);
            const double scale = (s > 0.0 && s > 1e-9 * fabs(mean[c])) ? s : 1.0;
            const int k = c < 3 ? c : 6 + (c - 3);
            nm[k] = (float)mean[c];
            nm[k + 3] = (float)scale;
        }
        for (int c = 0; c < 3; ++c) {
            norm->in_mean[c] = nm[c];
            norm->in_scale[c] = nm[3 + c];
            norm->out_mean[c] = nm[6 + c];
            norm->out_scale[c] = nm[9 + c];
        }
    }
    __syncthreads();
    for (int i = t; i < n; i += kPrepThreads)
        for (int c = 0; c < 3; ++c) {
            x[3 * i + c] = (input_feature(x[3 * i + c], c) - nm[c]) / nm[3 + c];
            const float yv = y[3 * i + c];
            const float tv = c == 1 ? yv : logf(yv);
            y[3 * i + c] = (tv - nm[6 + c]) / nm[9 + c];
        }
}

// ---------------------------------------------------------------------------------
// Forward + backward. Tiles of 16 samples, in blocks of 256 threads:
//   SPLIT = 1: CTA b takes tiles b, b + gridDim.x, ... and keeps the gradient entries it owns in
//     registers: gW2: 16 per thread (k = t & 63, j = 16 (t >> 6) + q), gb2: threads 0..63,
//     gW3 / gb3: threads 0..191 / 192..194, gW1 / gb1: 0..191 / 192..255.
//   SPLIT = 4: cluster b takes tile b. Each of its CTAs carries four samples forward and back and
//     sends the others what they need of it through distributed shared memory; then CTA r sums
//     the gradient entries of hidden units 16 r .. 16 r + 15 over the tile's 16 samples.
// Activations of a tile live in shared memory; dz overwrites z in place.
// What bounds it: the chain load weights -> layer -> layer -> back, once per tile, not the
// arithmetic (14 MFLOP at 512 samples): so four CTAs share a tile while they all are resident,
// kMaxGradCtas in all. Every sum runs in the order of the samples and of the tiles, however
// they are split: weights are used rounded to BF16, so a gradient off by one rounding sends
// some weight to the other neighbour at some step, and with tiles of 4 samples two of three runs
// of 50 steps ended 3e-5 away from the others. Rows of W2 are padded to 68 floats: 16-byte row
// reads (forward) and column reads (backward) are both free of bank conflicts. 50 Adam steps at
// 512 samples (both kernels, the call included): 520 us, against 1465 us with one CTA per
// tile, a serial partial sum and no launch overlap.
// ---------------------------------------------------------------------------------
__device__ __forceinline__ void grid_dependency_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void grid_dependents_launch() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// address of the same shared-memory variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t in_cta(const void *p, unsigned rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void store_cta(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// what a CTA of a cluster sums over the tile's samples: a_1 and, of its own 16 hidden units, a_2,
// dz_2 and dz_1; inputs, residuals and their scaled form
struct TileShare {
    __align__(16) float a1[kTile * H];
    float a2[kTile * 16], dz2[kTile * 16], dz1[kTile * 16];
    float x[kTile * IN], dout[kTile * OUT], res[kTile * OUT];
};

template <int SPLIT>
__global__ void __launch_bounds__(kThreads, 2)
k_mlp_grad(const __nv_bfloat16 *__restrict__ wbf, const float *__restrict__ xn,
           const float *__restrict__ tn, MlpState *__restrict__ st, int bump_step,
           float *__restrict__ part, float *__restrict__ lpart) {
    constexpr int TILE = kTile / SPLIT;   // samples of the CTA
    constexpr int NQ = TILE / 4;          // samples per thread in the hidden layers
    constexpr bool CL = SPLIT > 1;
    struct None {};
    __shared__ SmemW w;
    __shared__ float sx[TILE * IN], dout[TILE * OUT], res[TILE * OUT];
    __shared__ __align__(16) float z1[TILE * H], a1[TILE * H], z2[TILE * H], a2[TILE * H];
    __shared__ std::conditional_t<CL, TileShare, None> sh;
    const int t = threadIdx.x;
    const unsigned rank = CL ? cluster_rank() : 0;
    const int tile0 = blockIdx.x / SPLIT, tiles = gridDim.x / SPLIT;
    if constexpr (CL) cluster_arrive();   // (waited for before the first store to another CTA)
    // the weights are the previous kernel's: wait for it (programmatic dependent launch)
    grid_dependency_wait();
    grid_dependents_launch();
    const int n = st->n;
    if (bump_step && blockIdx.x == 0 && t == 0) {
        st->step += 1;
        st->pow1 *= (double)st->beta1;
        st->pow2 *= (double)st->beta2;
    }
    load_weights(w, wbf);
    const float dscale = 2.0f / (3.0f * (float)n);

    float gw2[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) gw2[q] = 0.f;
    float gb2 = 0.f, g3 = 0.f, g1 = 0.f, lsum = 0.f;

    const int jj = t & 63, sg = t >> 6;   // unit and sample group (uniform in a warp)
    for (int base = tile0 * kTile + (int)rank * TILE; base < n || CL; base += tiles * kTile) {
        __syncthreads();   // weights loaded / previous tile consumed
        if (t < TILE * IN) sx[t] = base + t / IN < n ? xn[(size_t)base * IN + t] : 0.f;
        __syncthreads();
        // layer 1
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int s = sg + 4 * q;
            float z = w.b1[jj];
#pragma unroll
            for (int i = 0; i < IN; ++i) z = fmaf(w.w1[jj * IN + i], sx[s * IN + i], z);
            z1[s * H + jj] = z;
            a1[s * H + jj] = gelu(z);
        }
        __syncthreads();
        if constexpr (CL) {
            cluster_wait();               // the others have started
            const int s = (int)rank * TILE + sg;
            const float v = a1[sg * H + jj];
#pragma unroll
            for (int c = 0; c < SPLIT; ++c) store_cta(in_cta(&sh.a1[s * H + jj], c), v);
            if (t < TILE * IN)
#pragma unroll
                for (int c = 0; c < SPLIT; ++c) store_cta(in_cta(&sh.x[(int)rank * TILE * IN + t], c), sx[t]);
        }
        // layer 2
        {
            float acc[NQ];
#pragma unroll
            for (int q = 0; q < NQ; ++q) acc[q] = w.b2[jj];
#pragma unroll 4
            for (int k = 0; k < H; k += 4) {
                const float4 wv = *reinterpret_cast<const float4 *>(&w.w2[jj * kW2Pitch + k]);
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const float4 av = *reinterpret_cast<const float4 *>(&a1[(sg + 4 * q) * H + k]);
                    acc[q] = fmaf(wv.x, av.x, acc[q]);
                    acc[q] = fmaf(wv.y, av.y, acc[q]);
                    acc[q] = fmaf(wv.z, av.z, acc[q]);
                    acc[q] = fmaf(wv.w, av.w, acc[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                z2[(sg + 4 * q) * H + jj] = acc[q];
                const float g = gelu(acc[q]);
                a2[(sg + 4 * q) * H + jj] = g;
                if constexpr (CL)
                    store_cta(in_cta(&sh.a2[((int)rank * TILE + sg) * 16 + (jj & 15)], jj >> 4), g);
            }
        }
        __syncthreads();
        // output layer and loss residual
        if (t < TILE * OUT) {
            const int s = t / OUT, c = t % OUT;
            const float target = base + s < n ? tn[(size_t)base * OUT + t] : 0.f;
            float o = w.b3[c];
#pragma unroll
            for (int k = 0; k < H; k += 4) {
                const float4 wv = *reinterpret_cast<const float4 *>(&w.w3[c * H + k]);
                const float4 av = *reinterpret_cast<const float4 *>(&a2[s * H + k]);
                o = fmaf(wv.x, av.x, o);
                o = fmaf(wv.y, av.y, o);
                o = fmaf(wv.z, av.z, o);
                o = fmaf(wv.w, av.w, o);
            }
            const float r = base + s < n ? o - target : 0.f;
            dout[t] = r * dscale;
            res[t] = r;
            if constexpr (CL) {
#pragma unroll
                for (int d = 0; d < SPLIT; ++d) store_cta(in_cta(&sh.dout[(int)rank * TILE * OUT + t], d), r * dscale);
                store_cta(in_cta(&sh.res[(int)rank * TILE * OUT + t], 0), r);
            }
        }
        __syncthreads();
        // gW3, gb3, loss; dz2 = (dout W3) * gelu'(z2) in place
        if constexpr (!CL) {
            if (t < OUT * H) {
                const int c = t >> 6, k = t & 63;
#pragma unroll
                for (int s = 0; s < TILE; ++s) g3 = fmaf(dout[s * OUT + c], a2[s * H + k], g3);
            } else if (t < OUT * H + OUT) {
                const int c = t - OUT * H;
                for (int s = 0; s < TILE; ++s) g3 += dout[s * OUT + c];
            } else if (t == kThreads - 1) {
                for (int k = 0; k < TILE * OUT; ++k) lsum = fmaf(res[k], res[k], lsum);
            }
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int s = sg + 4 * q;
            float d = 0.f;
#pragma unroll
            for (int c = 0; c < OUT; ++c) d = fmaf(dout[s * OUT + c], w.w3[c * H + jj], d);
            d = d * gelu_grad(z2[s * H + jj]);
            z2[s * H + jj] = d;
            if constexpr (CL)
                store_cta(in_cta(&sh.dz2[((int)rank * TILE + sg) * 16 + (jj & 15)], jj >> 4), d);
        }
        __syncthreads();
        // gW2, gb2; dz1 = (dz2 W2) * gelu'(z1) in place
        if constexpr (!CL) {
#pragma unroll 4
            for (int s = 0; s < TILE; ++s) {
                const float av = a1[s * H + jj];
#pragma unroll
                for (int q = 0; q < 16; q += 4) {
                    const float4 d = *reinterpret_cast<const float4 *>(&z2[s * H + 16 * sg + q]);
                    gw2[q] = fmaf(d.x, av, gw2[q]);
                    gw2[q + 1] = fmaf(d.y, av, gw2[q + 1]);
                    gw2[q + 2] = fmaf(d.z, av, gw2[q + 2]);
                    gw2[q + 3] = fmaf(d.w, av, gw2[q + 3]);
                }
            }
            if (t < H)
                for (int s = 0; s < TILE; ++s) gb2 += z2[s * H + t];
        }
        {
            float acc[NQ];
#pragma unroll
            for (int q = 0; q < NQ; ++q) acc[q] = 0.f;
#pragma unroll 4
            for (int j = 0; j < H; j += 4) {
                float wv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) wv[e] = w.w2[(j + e) * kW2Pitch + jj];
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const float4 d = *reinterpret_cast<const float4 *>(&z2[(sg + 4 * q) * H + j]);
                    acc[q] = fmaf(d.x, wv[0], acc[q]);
                    acc[q] = fmaf(d.y, wv[1], acc[q]);
                    acc[q] = fmaf(d.z, wv[2], acc[q]);
                    acc[q] = fmaf(d.w, wv[3], acc[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int s = sg + 4 * q;
                const float d = acc[q] * gelu_grad(z1[s * H + jj]);
                if constexpr (CL)
                    store_cta(in_cta(&sh.dz1[((int)rank * TILE + sg) * 16 + (jj & 15)], jj >> 4), d);
                else
                    z1[s * H + jj] = d;
            }
        }
        if constexpr (CL) break;
        __syncthreads();
        // gW1, gb1
        if (t < H * IN) {
            const int j = t / IN, i = t % IN;
#pragma unroll
            for (int s = 0; s < TILE; ++s) g1 = fmaf(z1[s * H + j], sx[s * IN + i], g1);
        } else {
            const int j = t - H * IN;
#pragma unroll
            for (int s = 0; s < TILE; ++s) g1 += z1[s * H + j];
        }
    }
    float *out = part + (size_t)tile0 * NP;
    if constexpr (CL) {
        cluster_arrive();
        cluster_wait();                   // the tile's samples are here; nothing is sent any more
        const int j = t >> 4, k = t & 15, u = 16 * (int)rank;
        // first the entries that a warp or two own, while the others go on to W2
        if (t >= 208) {
            if (t < 256) {                // gW3 of units u ..
                const int c = (t - 208) >> 4;
#pragma unroll
                for (int s = 0; s < kTile; ++s) g3 = fmaf(sh.dout[s * OUT + c], sh.a2[s * 16 + k], g3);
                out[OW3 + c * H + u + k] = g3;
            }
        } else if (t >= 160) {            // gW1 of units u ..
            const int e = t - 160;
#pragma unroll
            for (int s = 0; s < kTile; ++s) g1 = fmaf(sh.dz1[s * 16 + e / IN], sh.x[s * IN + e % IN], g1);
            out[OW1 + u * IN + e] = g1;
        } else if (t >= 128) {            // gb1, gb2
            const float *d = t < 144 ? sh.dz1 : sh.dz2;
#pragma unroll
            for (int s = 0; s < kTile; ++s) gb2 += d[s * 16 + k];
            out[(t < 144 ? OB1 : OB2) + u + k] = gb2;
        } else if (t >= 96 && t < 96 + OUT && rank == 0) {
#pragma unroll
            for (int s = 0; s < kTile; ++s) g3 += sh.dout[s * OUT + t - 96];
            out[OB3 + t - 96] = g3;
        } else if (t == 64 && rank == 0) {
#pragma unroll
            for (int e = 0; e < kTile * OUT; ++e) lsum = fmaf(sh.res[e], sh.res[e], lsum);
            lpart[tile0] = lsum;
        }
#pragma unroll
        for (int s = 0; s < kTile; ++s) {
            const float d = sh.dz2[s * 16 + j];
#pragma unroll
            for (int q = 0; q < 4; ++q) gw2[q] = fmaf(d, sh.a1[s * H + 16 * q + k], gw2[q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) out[OW2 + (u + j) * H + 16 * q + k] = gw2[q];
    } else {
#pragma unroll
        for (int q = 0; q < 16; ++q) out[OW2 + (16 * sg + q) * H + jj] = gw2[q];
        if (t < H) out[OB2 + t] = gb2;
        if (t < OUT * H) out[OW3 + t] = g3;
        else if (t < OUT * H + OUT) out[OB3 + t - OUT * H] = g3;
        if (t < H * IN) out[OW1 + t] = g1;
        else out[OB1 + t - H * IN] = g1;
        if (t == kThreads - 1) lpart[tile0] = lsum;
    }
}

// Sum of the partial gradients in the order of the tiles, then Adam on the FP32 master copy. A
// CTA owns 32 parameters: its warps fetch the partials into shared memory (128-byte reads,
// several in flight), then one warp adds them; the bias corrections come from the running powers
// of beta1 and beta2 that k_mlp_grad advances in FP64. One thread per parameter with a serial
// sum of 32 partials and two FP64 pow took 17.6 us at 512 samples.
constexpr int kAdamThreads = 256, kAdamParams = 32;

__global__ void __launch_bounds__(kAdamThreads)
k_mlp_adam(const float *__restrict__ part, const float *__restrict__ lpart, int nparts,
           MlpState *__restrict__ st, float *__restrict__ master, float *__restrict__ m1,
           float *__restrict__ m2, __nv_bfloat16 *__restrict__ wbf, float *__restrict__ grad_out) {
    constexpr int NW = kAdamThreads / 32;
    __shared__ float parts[kMaxGradCtas][kAdamParams];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = blockIdx.x * kAdamParams + lane;
    grid_dependency_wait();
    grid_dependents_launch();
    if (p < NP) {
#pragma unroll 8
        for (int c = warp; c < nparts; c += NW) parts[c][lane] = part[(size_t)c * NP + p];
    }
    __syncthreads();
    if (blockIdx.x == 0 && warp == 1) {   // the loss: lanes take every 32nd partial, then a butterfly
        double l = 0.0;
        for (int c = lane; c < nparts; c += 32) l += (double)lpart[c];
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) l += __shfl_xor_sync(0xffffffffu, l, m);
        if (lane == 0) st->loss = (float)(l / (3.0 * st->n));
    }
    if (warp != 0 || p >= NP) return;
    float g = 0.f;
#pragma unroll 16
    for (int c = 0; c < nparts; ++c) g += parts[c][lane];
    if (grad_out) {   // gradient only (no update)
        grad_out[p] = g;
        return;
    }
    const float b1 = st->beta1, b2 = st->beta2;
    const float m = fmaf(b1, m1[p], (1.f - b1) * g);
    const float v = fmaf(b2, m2[p], (1.f - b2) * g * g);
    m1[p] = m;
    m2[p] = v;
    const float c1 = (float)(1.0 - st->pow1);
    const float c2 = (float)(1.0 - st->pow2);
    const float upd = st->lr * (m / c1) / (sqrtf(v / c2) + st->eps);
    const float th = master[p] - upd;
    master[p] = th;
    wbf[p] = __float2bfloat16_rn(th);
}

__global__ void k_mlp_refresh_bf16(const float *__restrict__ master, __nv_bfloat16 *__restrict__ wbf) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < NP) wbf[p] = __float2bfloat16_rn(master[p]);
}

// ---------------------------------------------------------------------------------
// Inference. A warp carries Q samples at a time; lane l owns hidden units 2l and 2l + 1 of
// both layers and keeps their W2 rows in registers as unit pairs, so the 64 x 64 layer is 64
// packed multiply-adds per lane and sample, each lane's sum in the order of k. The layer's
// inputs go round the warp through shared memory, every activation stored twice (a, a) so
// that one 16-byte broadcast load feeds two packed multiply-adds. The output sums are a
// fixed butterfly over the lanes.
// What bounds it: the serial chain of one evaluation (two erf-based activations and a
// 64-long sum), times 42 evaluations for the inversion. One thread per sample (weights re-read
// from shared memory) took 2346 us for 4097 inversions and as long for 24, 33 CTAs busy; a
// warp per sample shortens the chain by 30 and fills the chip: lb_mlp_forward and
// lb_mlp_invert_kappa of 4097 samples, copies included, 181 us against 2449 us (153 us without
// the halvings that change nothing).
// ---------------------------------------------------------------------------------
constexpr int kInferThreads = 128, kInferWarps = kInferThreads / 32;
constexpr int kInferCtas = 2;      // resident CTAs per SM (the weights take 128 registers a thread)

struct LaneWeights {
    float2 w2[H];                  // (W2[2l][k], W2[2l+1][k])
    float2 w1[IN], b1, b2;
};

__device__ __forceinline__ float2 bf16_pair(const __nv_bfloat16 *__restrict__ w, int i, int j) {
    return make_float2(__bfloat162float(w[i]), __bfloat162float(w[j]));
}

__device__ __forceinline__ void load_lane_weights(LaneWeights &L, const __nv_bfloat16 *__restrict__ w) {
    const int j = 2 * (threadIdx.x & 31);
    const uint4 *r0 = reinterpret_cast<const uint4 *>(w + OW2 + j * H);   // 16-byte aligned rows
    const uint4 *r1 = reinterpret_cast<const uint4 *>(w + OW2 + (j + 1) * H);
#pragma unroll
    for (int c = 0; c < H / 8; ++c) {
        const uint4 u = r0[c], v = r1[c];
        const unsigned a[4] = {u.x, u.y, u.z, u.w}, b[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            L.w2[8 * c + 2 * e] = make_float2(__uint_as_float(a[e] << 16), __uint_as_float(b[e] << 16));
            L.w2[8 * c + 2 * e + 1] = make_float2(__uint_as_float(a[e] & 0xffff0000u),
                                                  __uint_as_float(b[e] & 0xffff0000u));
        }
    }
#pragma unroll
    for (int i = 0; i < IN; ++i) L.w1[i] = bf16_pair(w, OW1 + j * IN + i, OW1 + (j + 1) * IN + i);
    L.b1 = bf16_pair(w, OB1 + j, OB1 + j + 1);
    L.b2 = bf16_pair(w, OB2 + j, OB2 + j + 1);
}
static_assert((OW2 * 2) % 16 == 0 && (H * 2) % 16 == 0, "W2 rows are read in 16-byte words");

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// second-layer activations of the lane's two units for Q standardised samples
template <int Q>
__device__ __forceinline__ void hidden_units(const LaneWeights &L, const float (&xs)[Q][IN],
                                             float4 (*act)[H / 2], float2 (&g)[Q]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        float2 z = L.b1;
#pragma unroll
        for (int i = 0; i < IN; ++i) z = fma2(L.w1[i], make_float2(xs[q][i], xs[q][i]), z);
        const float a0 = gelu(z.x), a1 = gelu(z.y);
        act[q][lane] = make_float4(a0, a0, a1, a1);
    }
    __syncwarp();
    float2 z[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) z[q] = L.b2;
#pragma unroll
    for (int k = 0; k < H / 2; ++k) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float4 a = act[q][k];
            z[q] = fma2(L.w2[2 * k], make_float2(a.x, a.y), z[q]);
            z[q] = fma2(L.w2[2 * k + 1], make_float2(a.z, a.w), z[q]);
        }
    }
    __syncwarp();                  // the activations are read: the next call may overwrite them
#pragma unroll
    for (int q = 0; q < Q; ++q) g[q] = make_float2(gelu(z[q].x), gelu(z[q].y));
}

__device__ __forceinline__ void standardise(const MlpNorm &nm, const float (&x)[3], float (&xs)[3]) {
#pragma unroll
    for (int i = 0; i < IN; ++i) xs[i] = (input_feature(x[i], i) - nm.in_mean[i]) / nm.in_scale[i];
}

__device__ __forceinline__ float sigma_of(const MlpNorm &nm, float o0) {
    return expf(fmaf(o0, nm.out_scale[0], nm.out_mean[0]));
}

template <int Q>
__global__ void __launch_bounds__(kInferThreads, kInferCtas)
k_mlp_forward(const __nv_bfloat16 *__restrict__ wbf, const MlpNorm *__restrict__ norm,
              const float *__restrict__ x, float *__restrict__ y, int n) {
    __shared__ float4 act[kInferWarps][Q][H / 2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    LaneWeights L;
    load_lane_weights(L, wbf);
    float2 w3[OUT];
    float b3[OUT];
#pragma unroll
    for (int c = 0; c < OUT; ++c) {
        w3[c] = bf16_pair(wbf, OW3 + c * H + 2 * lane, OW3 + c * H + 2 * lane + 1);
        b3[c] = __bfloat162float(wbf[OB3 + c]);
    }
    const MlpNorm nm = *norm;
    for (int i = (blockIdx.x * kInferWarps + warp) * Q; i < n; i += gridDim.x * kInferWarps * Q) {
        float xs[Q][IN];
        float2 g[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int s = min(i + q, n - 1);   // a ragged last group repeats its last sample
            const float xv[3] = {x[3 * s], x[3 * s + 1], x[3 * s + 2]};
            standardise(nm, xv, xs[q]);
        }
        hidden_units<Q>(L, xs, act[warp], g);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            float o[OUT];
#pragma unroll
            for (int c = 0; c < OUT; ++c) o[c] = output_unit(w3[c], b3[c], g[q]);
            if (lane == 0 && i + q < n) {
                y[3 * (i + q) + 0] = sigma_of(nm, o[0]);
                y[3 * (i + q) + 1] = fmaf(o[1], nm.out_scale[1], nm.out_mean[1]);
                y[3 * (i + q) + 2] = expf(fmaf(o[2], nm.out_scale[2], nm.out_mean[2]));
            }
        }
    }
}

template <int Q>
__global__ void __launch_bounds__(kInferThreads, kInferCtas)
k_mlp_invert(const __nv_bfloat16 *__restrict__ wbf, const MlpNorm *__restrict__ norm,
             const float *__restrict__ qs, int n, float lo0, float hi0, float *__restrict__ kappa) {
    __shared__ float4 act[kInferWarps][Q][H / 2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    LaneWeights L;
    load_lane_weights(L, wbf);
    const float2 w3 = bf16_pair(wbf, OW3 + 2 * lane, OW3 + 2 * lane + 1);
    const float b3 = __bfloat162float(wbf[OB3]);
    const MlpNorm nm = *norm;
    for (int i = (blockIdx.x * kInferWarps + warp) * Q; i < n; i += gridDim.x * kInferWarps * Q) {
        float xs[Q][IN], lo[Q], hi[Q], target[Q];
        bool ok[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int s = min(i + q, n - 1);   // a ragged last group repeats its last query
            const float xv[3] = {qs[3 * s], 0.f, qs[3 * s + 1]};
            standardise(nm, xv, xs[q]);        // T/T_c and tau_v stay through the bisection
            target[q] = qs[3 * s + 2];
            lo[q] = lo0;
            hi[q] = hi0;
            ok[q] = true;
        }
        // one call site of the network (the bracket check is iterations -2 and -1)
#pragma unroll 1
        for (int it = -2; it < kBisect; ++it) {
            float k[Q];
            float2 g[Q];
            bool any = false;          // a query that is still being bisected
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                k[q] = it == -2 ? lo[q] : (it == -1 ? hi[q] : 0.5f * (lo[q] + hi[q]));
                xs[q][1] = (input_feature(k[q], 1) - nm.in_mean[1]) / nm.in_scale[1];
            }
            hidden_units<Q>(L, xs, act[warp], g);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const float s = sigma_of(nm, output_unit(w3, b3, g[q]));
                if (it < 0) {
                    ok[q] = it == -2 ? s >= target[q] : ok[q] && s <= target[q];
                    any |= ok[q];
                } else {
                    // a halving that moves neither end (the ends are adjacent floats after 24 to
                    // 30 of them) would be followed by the same one: the rest is left out
                    float &end = s > target[q] ? lo[q] : hi[q];
                    any |= ok[q] && end != k[q];
                    end = k[q];
                }
            }
            if (!any) break;                   // the same in every lane
        }
#pragma unroll
        for (int q = 0; q < Q; ++q)
            if (lane == 0 && i + q < n)
                kappa[i + q] = ok[q] ? 0.5f * (lo[q] + hi[q]) : __int_as_float(0x7fc00000);
    }
}

// Samples per warp and grid for n samples: one per warp while every sample finds a resident
// warp (the chain of one sample is then all there is), else two (their chains overlap and
// share the weights' registers); the grid is at most the resident CTAs, which walk on.
struct InferLaunch {
    int q, grid;
};

InferLaunch infer_launch(int sms, int n) {
    InferLaunch l;
    l.q = n <= sms * kInferCtas * kInferWarps ? 1 : 2;
    const int per_cta = kInferWarps * l.q;
    l.grid = std::min((n + per_cta - 1) / per_cta, sms * kInferCtas);
    return l;
}

}  // namespace

struct lb_mlp {
    cudaStream_t stream = nullptr;
    int max_samples = 0, n = 0;
    int parts = 0, split = 1;     // partial gradients, CTAs that share one (k_mlp_grad)
    int sms = 1;
    float *master = nullptr, *m1 = nullptr, *m2 = nullptr, *xn = nullptr, *tn = nullptr;
    float *part = nullptr, *lpart = nullptr, *grad = nullptr;
    __nv_bfloat16 *wbf = nullptr;
    MlpNorm *norm = nullptr;
    MlpState *st = nullptr;
    float *io = nullptr;          // staging for forward / invert
    size_t io_floats = 0;
    long long steps = 0;
    bool have_norm = false;
    cudaGraphExec_t graph = nullptr;
    std::string msg;
};

namespace {

lb_status mfail(lb_mlp *m, lb_status s, const std::string &msg) {
    if (m) m->msg = msg;
    return lbm::reported(s);
}

#define LB_MCUDA(m, call)                                                              \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess)                                                         \
            return mfail((m), LB_ECUDA, std::string(#call ": ") + cudaGetErrorString(e_)); \
    } while (0)

bool finite3(const float *v) {
    return std::isfinite(v[0]) && std::isfinite(v[1]) && std::isfinite(v[2]);
}

// launch with programmatic dependent launch: the kernel's set-up overlaps the previous
// kernel's end, it waits (griddepcontrol.wait) before its first access to global memory
template <typename K, typename... A>
cudaError_t launch_dependent(K kern, int grid, int block, int cluster, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// CTAs per tile for n samples (see k_mlp_grad)
int split_for(int n) { return n <= kTile * (kMaxGradCtas / kSplit) ? kSplit : 1; }

cudaError_t launch_grad(lb_mlp *m, int bump, cudaStream_t s) {
    return launch_dependent(m->split == kSplit ? k_mlp_grad<kSplit> : k_mlp_grad<1>, m->parts * m->split, kThreads,
                            m->split, s, (const __nv_bfloat16 *)m->wbf, (const float *)m->xn,
                            (const float *)m->tn, m->st, bump, m->part, m->lpart);
}

cudaError_t launch_adam(lb_mlp *m, float *grad_out, cudaStream_t s) {
    return launch_dependent(k_mlp_adam, (NP + kAdamParams - 1) / kAdamParams, kAdamThreads, 1, s,
                            (const float *)m->part, (const float *)m->lpart, m->parts, m->st,
                            m->master, m->m1, m->m2, m->wbf, grad_out);
}

lb_status ensure_graph(lb_mlp *m) {
    if (m->graph) return LB_OK;
    cudaStream_t cap = nullptr;
    LB_MCUDA(m, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        for (int i = 0; i < kGraphSteps && e == cudaSuccess; ++i) {
            e = launch_grad(m, 1, cap);
            if (e == cudaSuccess) e = launch_adam(m, nullptr, cap);
        }
        cudaError_t e2 = cudaStreamEndCapture(cap, &g);
        if (e == cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&m->graph, g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cap);
    if (e != cudaSuccess)
        return mfail(m, LB_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
    return LB_OK;
}

void drop_graph(lb_mlp *m) {
    if (m->graph) cudaGraphExecDestroy(m->graph);
    m->graph = nullptr;
}

lb_status ensure_io(lb_mlp *m, size_t floats) {
    if (floats <= m->io_floats) return LB_OK;
    if (m->io) cudaFree(m->io);
    m->io = nullptr;
    m->io_floats = 0;
    if (cudaMalloc(&m->io, floats * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        return mfail(m, LB_ENOMEM, "staging allocation failed");
    }
    m->io_floats = floats;
    return LB_OK;
}

}  // namespace

extern "C" {

lb_status lb_mlp_create(lb_mlp **out, int max_samples, void *stream) {
    if (!out) return LB_EINVAL;
    *out = nullptr;
    if (max_samples < 1 || max_samples > kMaxSamples) return LB_EINVAL;
    lb_mlp *m = new (std::nothrow) lb_mlp();
    if (!m) return LB_ENOMEM;
    m->stream = static_cast<cudaStream_t>(stream);
    m->max_samples = max_samples;
    const size_t ns = (size_t)max_samples;
    int dev = 0;
    bool ok = cudaGetDevice(&dev) == cudaSuccess &&
              cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
              cudaMalloc(&m->master, NP * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->m1, NP * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->m2, NP * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->grad, NP * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->wbf, NP * sizeof(__nv_bfloat16)) == cudaSuccess &&
              cudaMalloc(&m->xn, ns * IN * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->tn, ns * OUT * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->part, (size_t)kMaxGradCtas * NP * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->lpart, kMaxGradCtas * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->norm, sizeof(MlpNorm)) == cudaSuccess &&
              cudaMalloc(&m->st, sizeof(MlpState)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        lb_mlp_free(m);
        return LB_ENOMEM;
    }
    std::vector<float> zero(NP, 0.f);
    if (lb_mlp_set_params(m, zero.data()) != LB_OK) {
        lb_mlp_free(m);
        return LB_ECUDA;
    }
    MlpNorm nm;
    for (int c = 0; c < 3; ++c) {
        nm.in_mean[c] = nm.out_mean[c] = 0.f;
        nm.in_scale[c] = nm.out_scale[c] = 1.f;
    }
    MlpState st{};
    if (cudaMemcpy(m->norm, &nm, sizeof nm, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(m->st, &st, sizeof st, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        lb_mlp_free(m);
        return LB_ECUDA;
    }
    *out = m;
    return LB_OK;
}

lb_status lb_mlp_set_params(lb_mlp *m, const float *params) {
    if (!m || !params) return LB_EINVAL;
    for (int p = 0; p < NP; ++p)
        if (!std::isfinite(params[p])) return mfail(m, LB_EINVAL, "non-finite parameter");
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    LB_MCUDA(m, cudaMemcpy(m->master, params, NP * sizeof(float), cudaMemcpyHostToDevice));
    LB_MCUDA(m, cudaMemset(m->m1, 0, NP * sizeof(float)));
    LB_MCUDA(m, cudaMemset(m->m2, 0, NP * sizeof(float)));
    LB_MCUDA(m, cudaMemset(m->st, 0, sizeof(int)));   // Adam step count
    k_mlp_refresh_bf16<<<(NP + 255) / 256, 256, 0, m->stream>>>(m->master, m->wbf);
    LB_MCUDA(m, cudaGetLastError());
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    m->steps = 0;
    return LB_OK;
}

lb_status lb_mlp_get_params(lb_mlp *m, float *params) {
    if (!m || !params) return LB_EINVAL;
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    LB_MCUDA(m, cudaMemcpy(params, m->master, NP * sizeof(float), cudaMemcpyDeviceToHost));
    return LB_OK;
}

lb_status lb_mlp_set_data(lb_mlp *m, const float *x, const float *y, int n) {
    if (!m || !x || !y) return LB_EINVAL;
    if (n < 1 || n > m->max_samples)
        return mfail(m, LB_EINVAL, "sample count outside [1, max_samples]");
    for (int i = 0; i < n; ++i) {
        if (!finite3(x + 3 * i) || !finite3(y + 3 * i))
            return mfail(m, LB_EINVAL, "non-finite sample " + std::to_string(i));
        if (!(y[3 * i] > 0.f && y[3 * i + 1] > 0.f && y[3 * i + 2] > 0.f))
            return mfail(m, LB_EINVAL, "target <= 0 in sample " + std::to_string(i));
        if (!(x[3 * i] < 1.f && x[3 * i + 1] < 1.f))
            return mfail(m, LB_EINVAL, "T/T_c or kappa >= 1 in sample " + std::to_string(i));
    }
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    LB_MCUDA(m, cudaMemcpy(m->xn, x, (size_t)n * IN * sizeof(float), cudaMemcpyHostToDevice));
    LB_MCUDA(m, cudaMemcpy(m->tn, y, (size_t)n * OUT * sizeof(float), cudaMemcpyHostToDevice));
    k_mlp_prepare<<<1, kPrepThreads, 0, m->stream>>>(m->xn, m->tn, n, m->norm);
    LB_MCUDA(m, cudaGetLastError());
    LB_MCUDA(m, cudaMemcpyAsync(&m->st->n, &n, sizeof(int), cudaMemcpyHostToDevice, m->stream));
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    m->n = n;
    const int split = split_for(n), parts = std::min((n + kTile - 1) / kTile, kMaxGradCtas);
    // the captured graph carries the grid and the kernel
    if (parts != m->parts || split != m->split) drop_graph(m);
    m->split = split;
    m->parts = parts;
    m->have_norm = true;
    return LB_OK;
}

lb_status lb_mlp_get_norm(lb_mlp *m, lb_mlp_norm *out) {
    if (!m || !out) return LB_EINVAL;
    MlpNorm nm;
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    LB_MCUDA(m, cudaMemcpy(&nm, m->norm, sizeof nm, cudaMemcpyDeviceToHost));
    static_assert(sizeof(MlpNorm) == sizeof(lb_mlp_norm), "norm layout");
    std::memcpy(out, &nm, sizeof nm);
    return LB_OK;
}

lb_status lb_mlp_set_norm(lb_mlp *m, const lb_mlp_norm *norm) {
    if (!m || !norm) return LB_EINVAL;
    for (int c = 0; c < 3; ++c)
        if (!(std::isfinite(norm->in_mean[c]) && std::isfinite(norm->out_mean[c]) &&
              norm->in_scale[c] > 0.f && std::isfinite(norm->in_scale[c]) &&
              norm->out_scale[c] > 0.f && std::isfinite(norm->out_scale[c])))
            return mfail(m, LB_EINVAL, "scales must be positive and finite");
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    LB_MCUDA(m, cudaMemcpy(m->norm, norm, sizeof(MlpNorm), cudaMemcpyHostToDevice));
    return LB_OK;
}

lb_status lb_mlp_loss_grad(lb_mlp *m, float *loss, float *grad) {
    if (!m) return LB_EINVAL;
    if (m->n < 1) return mfail(m, LB_EINVAL, "no training data");
    LB_MCUDA(m, launch_grad(m, 0, m->stream));
    LB_MCUDA(m, launch_adam(m, m->grad, m->stream));
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    if (grad) LB_MCUDA(m, cudaMemcpy(grad, m->grad, NP * sizeof(float), cudaMemcpyDeviceToHost));
    if (loss)
        LB_MCUDA(m, cudaMemcpy(loss, &m->st->loss, sizeof(float), cudaMemcpyDeviceToHost));
    return LB_OK;
}

lb_status lb_mlp_train(lb_mlp *m, int steps, float lr, float beta1, float beta2, float eps,
                       float *loss) {
    const lbm::NvtxRange nvtx_range("lb_mlp_train");
    if (!m || steps < 0) return LB_EINVAL;
    if (m->n < 1) return mfail(m, LB_EINVAL, "no training data");
    if (!(lr > 0.f && std::isfinite(lr) && beta1 >= 0.f && beta1 < 1.f && beta2 >= 0.f &&
          beta2 < 1.f && eps > 0.f && std::isfinite(eps)))
        return mfail(m, LB_EINVAL, "bad Adam hyper-parameters");
    const float hp[4] = {lr, beta1, beta2, eps};
    const double pw[2] = {std::pow((double)beta1, (double)m->steps),
                          std::pow((double)beta2, (double)m->steps)};
    LB_MCUDA(m, cudaMemcpyAsync(&m->st->lr, hp, sizeof hp, cudaMemcpyHostToDevice, m->stream));
    LB_MCUDA(m, cudaMemcpyAsync(&m->st->pow1, pw, sizeof pw, cudaMemcpyHostToDevice, m->stream));
    // the host arrays must stay valid until the copies ran
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    int left = steps;
    while (left >= kGraphSteps) {
        lb_status s = ensure_graph(m);
        if (s != LB_OK) return s;
        LB_MCUDA(m, cudaGraphLaunch(m->graph, m->stream));
        left -= kGraphSteps;
    }
    for (; left > 0; --left) {
        LB_MCUDA(m, launch_grad(m, 1, m->stream));
        LB_MCUDA(m, launch_adam(m, nullptr, m->stream));
    }
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    m->steps += steps;
    if (loss)
        LB_MCUDA(m, cudaMemcpy(loss, &m->st->loss, sizeof(float), cudaMemcpyDeviceToHost));
    return LB_OK;
}

long long lb_mlp_steps_done(const lb_mlp *m) { return m ? m->steps : -1; }

lb_status lb_mlp_forward(lb_mlp *m, const float *x, float *y, int n) {
    if (!m || n < 0 || n > kMaxForward || (n > 0 && (!x || !y))) return LB_EINVAL;
    if (n == 0) return LB_OK;
    for (int i = 0; i < n; ++i)
        if (!(finite3(x + 3 * i) && x[3 * i] < 1.f && x[3 * i + 1] < 1.f))
            return mfail(m, LB_EINVAL, "need finite inputs with T/T_c < 1 and kappa < 1");
    lb_status s = ensure_io(m, (size_t)n * 6);
    if (s != LB_OK) return s;
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    LB_MCUDA(m, cudaMemcpy(m->io, x, (size_t)n * 3 * sizeof(float), cudaMemcpyHostToDevice));
    const InferLaunch l = infer_launch(m->sms, n);
    (l.q == 1 ? k_mlp_forward<1> : k_mlp_forward<2>)<<<l.grid, kInferThreads, 0, m->stream>>>(
        m->wbf, m->norm, m->io, m->io + (size_t)n * 3, n);
    LB_MCUDA(m, cudaGetLastError());
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    LB_MCUDA(m, cudaMemcpy(y, m->io + (size_t)n * 3, (size_t)n * 3 * sizeof(float),
                           cudaMemcpyDeviceToHost));
    return LB_OK;
}

lb_status lb_mlp_invert_kappa(lb_mlp *m, const float *q, int n, float kappa_lo,
                              float kappa_hi, float *kappa) {
    if (!m || n < 0 || n > kMaxSamples || (n > 0 && (!q || !kappa))) return LB_EINVAL;
    if (!(std::isfinite(kappa_lo) && kappa_lo < kappa_hi && kappa_hi < 1.f))
        return mfail(m, LB_EINVAL, "need kappa_lo < kappa_hi < 1");
    if (n == 0) return LB_OK;
    for (int i = 0; i < n; ++i)
        if (!(finite3(q + 3 * i) && q[3 * i] < 1.f))
            return mfail(m, LB_EINVAL, "need finite queries with T/T_c < 1");
    lb_status s = ensure_io(m, (size_t)n * 4);
    if (s != LB_OK) return s;
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    LB_MCUDA(m, cudaMemcpy(m->io, q, (size_t)n * 3 * sizeof(float), cudaMemcpyHostToDevice));
    const InferLaunch l = infer_launch(m->sms, n);
    (l.q == 1 ? k_mlp_invert<1> : k_mlp_invert<2>)<<<l.grid, kInferThreads, 0, m->stream>>>(
        m->wbf, m->norm, m->io, n, kappa_lo, kappa_hi, m->io + (size_t)n * 3);
    LB_MCUDA(m, cudaGetLastError());
    LB_MCUDA(m, cudaStreamSynchronize(m->stream));
    LB_MCUDA(m, cudaMemcpy(kappa, m->io + (size_t)n * 3, (size_t)n * sizeof(float),
                           cudaMemcpyDeviceToHost));
    return LB_OK;
}

const char *lb_mlp_last_error(const lb_mlp *m) { return m ? m->msg.c_str() : "null network"; }

void lb_mlp_free(lb_mlp *m) {
    if (!m) return;
    cudaStreamSynchronize(m->stream);
    drop_graph(m);
    float *fl[] = {m->master, m->m1, m->m2, m->xn, m->tn, m->part, m->lpart, m->grad, m->io};
    for (float *p : fl)
        if (p) cudaFree(p);
    if (m->wbf) cudaFree(m->wbf);
    if (m->norm) cudaFree(m->norm);
    if (m->st) cudaFree(m->st);
    delete m;
}

}  // extern "C"
