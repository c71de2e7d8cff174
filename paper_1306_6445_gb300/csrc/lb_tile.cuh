// The tile kernels: no staging ring, one short dependent chain per step. FP32 and BF16 storage use
// one CTA per tile of 64 x R sites, which reads memory (k_tile_step, launch variant 7) or brings the
// tile into shared memory first (k_staged_tile_step, variant 8; k_batch_tile, the same for groups of
// lattices); FP64 uses a psi pass and a collision pass (k_psi_site, k_collide_site, variant 7), one
// site per thread. Same state
// layout, arithmetic and results, bit for bit, as the ring kernels of lb_step.cuh.
#pragma once

#include <algorithm>

#include "lb_step.cuh"

namespace lbm {

namespace {

// The planes of a buffer as uniform byte addresses; sites are 32-bit byte offsets from them, so
// a load or store takes one offset register and an immediate, no 64-bit address arithmetic.
template <typename T>
__device__ __forceinline__ const char *plane_bytes(const T *g, unsigned plane, int a) {
    return reinterpret_cast<const char *>(g) + (size_t)plane_of(a) * plane * sizeof(T);
}
template <typename T>
__device__ __forceinline__ T at_site(const char *pl, unsigned off, int dx) {
    return *reinterpret_cast<const T *>(pl + off + dx * (int)sizeof(T));
}
// the stored values of columns x + dx, x + dx + 1 (off: column x)
template <typename T>
__device__ __forceinline__ V2<Arith<T>> pair_at(const char *pl, unsigned off, int dx) {
    if (dx == 0) return ring_pair<T>(reinterpret_cast<const T *>(pl + off));
    return V2<Arith<T>>(stored_val<T>(at_site<T>(pl, off, dx)), stored_val<T>(at_site<T>(pl, off, dx + 1)));
}
// the stored values at columns offA + dx and offB + dx
template <typename T>
__device__ __forceinline__ V2<Arith<T>> two_at(const char *pl, unsigned offA, unsigned offB, int dx) {
    return V2<Arith<T>>(stored_val<T>(at_site<T>(pl, offA, dx)), stored_val<T>(at_site<T>(pl, offB, dx)));
}

// f pulled at a site pair: get(a, row, dx) returns stored population a of the row (0: the row
// below, 1: the row, 2: the row above) at column offset dx. bottom / top: the row is the
// lattice's first / last and BC has a boundary there.
template <int BC, typename A, typename F>
__device__ __forceinline__ void pull_rows(V2<A> (&f)[9], bool bottom, bool top, F get) {
    f[0] = get(0, 1, 0);
    f[1] = get(1, 1, -1);
    f[3] = get(3, 1, 1);
    if (BC != 0 && bottom) {          // bounced back from the wall below
        f[2] = get(4, 1, 0);
        f[5] = get(7, 1, 0);
        f[6] = get(8, 1, 0);
    } else {
        f[2] = get(2, 0, 0);
        f[5] = get(5, 0, -1);
        f[6] = get(6, 0, 1);
    }
    if (BC == 1 && top) {
        f[4] = get(2, 1, 0);
        f[7] = get(5, 1, 0);
        f[8] = get(6, 1, 0);
    } else if (BC == 2 && top) {      // open top: from the top row itself
        f[4] = get(4, 1, 0);
        f[7] = get(7, 1, 1);
        f[8] = get(8, 1, -1);
    } else {
        f[4] = get(4, 2, 0);
        f[7] = get(7, 2, 1);
        f[8] = get(8, 2, -1);
    }
}

constexpr int TILE_W = DIRECT_COLS;   // columns of a tile: one warp carries a row of it
constexpr int TILE_PW = TILE_W + 4;   // psi row: columns x0-2 .. x0+65

// The second half of a tile's step, after the barrier that completes psi: collide the warp's row
// (populations f of columns x, x + 1 of row y; psi rows y - 1 .. y + 1 in psis[warp] ..) and store.
template <typename T, int BC, bool SR, int ROWS, typename PT>
__device__ __forceinline__ void finish_tile(V2<Arith<T>> (&f)[9], const Arith<T> (&psis)[ROWS][TILE_PW],
                                            const PT &P, T *__restrict__ gout, const int x0,
                                            const int x, const int y, const int warp, const int w,
                                            const bool both, const int nx, const int ny,
                                            const int pitch, const unsigned plane) {
    using A = Arith<T>;
    const A *p0 = psis[warp + 1];
    const A *pm = (BC != 0 && y == 0) ? p0 : psis[warp];
    const A *pp = (BC != 0 && y == ny - 1) ? p0 : psis[warp + 2];
    const int c = x - x0 + 2;
    const V2<A> m0 = lds_pair<A>(pm + c), z0 = lds_pair<A>(p0 + c), q0 = lds_pair<A>(pp + c);
    V2<A> pn[9];
    pn[0] = z0;
    pn[1] = V2<A>(z0.hi(), p0[c + 2]);
    pn[2] = q0;
    pn[3] = V2<A>(p0[c - 1], z0.lo());
    pn[4] = m0;
    pn[5] = V2<A>(q0.hi(), pp[c + 2]);
    pn[6] = V2<A>(pp[c - 1], q0.lo());
    pn[7] = V2<A>(pm[c - 1], m0.lo());
    pn[8] = V2<A>(m0.hi(), pm[c + 2]);
    collide<A, BC == 2, std::is_same<T, __nv_bfloat16>::value>(f, pn, P);

    const unsigned rowi = (unsigned)y * (unsigned)pitch;
    const unsigned key = store_key<T, SR>(x, y, P);
    T *out = gout + rowi + (unsigned)(x + GH<T>);
    auto plane_at = [&](T *p, int a) { return p + (size_t)plane_of(a) * plane; };
    if (w == TILE_W) {                // a whole tile (CTA-uniform): every lane stores two sites
#pragma unroll
        for (int a = 0; a < 9; ++a)
            store_pop_pair<T, SR>(plane_at(out, a), f[a], true, store_bits<T, SR>(key, a));
    } else {
#pragma unroll
        for (int a = 0; a < 9; ++a)
            store_pop_pair<T, SR>(plane_at(out, a), f[a], both, store_bits<T, SR>(key, a));
    }
    if (x0 == 0 || x0 + TILE_W >= nx - 2) {   // CTA-uniform: a tile at a side of the lattice
        if (BC != 2 && (nx & 1) == 0) {
            // even width: the pairs (0, 1) and (nx-2, nx-1) have their images as pairs
            if (x == 0 || x == nx - 2) {
                T *img = x == 0 ? out + nx : out - nx;
#pragma unroll
                for (int a = 0; a < 9; ++a)
                    store_pop_pair<T, SR>(plane_at(img, a), f[a], true, store_bits<T, SR>(key, a));
            }
        } else {
            store_ghosts<T, BC, SR>(gout, f, x, rowi, nx, plane, both, key);
        }
    }
}

// resident CTAs the tile kernel is compiled for: 80 registers per thread (128 with the
// stochastic-rounding hash)
__host__ __device__ constexpr int tile_ctas(int R, bool sr) {
    return 65536 / (32 * R * (sr ? 128 : 80));
}

// One time step of a tile: columns x0 .. x0+63, rows y0 .. y0+R-1. Warp r pulls row y0 + r
// (two sites per lane, kept in registers) and forms its psi; warps 0 and 1 also form psi of
// the rows below and above the tile, warp 2 that of the two columns beside it. After one
// barrier every warp collides its row.
// What bounds it: the latency of one load -> psi -> barrier -> collide -> store chain where the
// lattice is small, issue where it fits in L2, memory beyond. Against the ring kernels it
// trades the serial march over rows (one barrier and one dependent shared-memory stage per
// row) and their per-row bookkeeping for 3 extra psi passes per 4 rows. Per step, against the
// ring kernel with the autotuner's launch: 64^2 2.3 / 9.4 us, 501 x 383 4.6 / 9.8, 600 x 225
// splash 4.1 / 12.8, 1024^2 12.0 / 15.1, 2048^2 51 / 49 (memory), BF16 stochastic 2048^2
// 61 / 65. Tiles of 3, 5, 6 and 8 rows were within 3 % of 4 or slower, as were 64 and 96
// registers.
template <typename T, int EOS, int BC, int R, bool SR, typename PT>
__device__ __forceinline__ void tile_step(const T *__restrict__ gin, T *__restrict__ gout,
                                          const PT &P, const int nx, const int ny,
                                          const int pitch, const unsigned plane, const int x0,
                                          const int y0, Arith<T> (&psis)[R + 2][TILE_PW],
                                          int *__restrict__ err) {
    static_assert(R >= 3, "three warps carry the rim");
    using A = Arith<T>;
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int w = min(TILE_W, nx - x0), n = min(R, ny - y0);
    const int y = y0 + warp, c0 = 2 * lane, x = x0 + c0;
    const bool act = warp < n && c0 < w, both = c0 + 1 < w;

    // byte offset of column 0 of row yy: periodic wrap, or the nearest row beyond a wall or an
    // open top (a wall link does not read it)
    auto row_at = [&](int yy) -> unsigned {
        if (BC == 0) yy = yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy);
        else yy = yy < 0 ? 0 : (yy >= ny ? ny - 1 : yy);
        return ((unsigned)yy * (unsigned)pitch + (unsigned)GH<T>) * (unsigned)sizeof(T);
    };
    const unsigned xo = (unsigned)x * (unsigned)sizeof(T);

    grid_dependency_wait();           // the previous step's state (programmatic dependent launch)
    grid_dependents_launch();

    V2<A> f[9];
    bool bad = false;
    if (act) {
        const unsigned o[3] = {row_at(y - 1) + xo, row_at(y) + xo, row_at(y + 1) + xo};
        pull_rows<BC, A>(f, y == 0, y == ny - 1, [&](int a, int r, int dx) {
            return pair_at<T>(plane_bytes(gin, plane, a), o[r], dx);
        });
    }
    if (warp < 3) {
        // the rim: a row below or above the tile (warps 0, 1) or the two columns beside it
        // (warp 2, one row per lane)
        const int yr = warp == 0 ? y0 - 1 : warp == 1 ? y0 + n : y0 - 1 + lane;
        const bool in = BC == 0 || (yr >= 0 && yr < ny);     // else psi is the edge row's
        const int yw = BC == 0 ? (yr < 0 ? yr + ny : (yr >= ny ? yr - ny : yr)) : yr;
        if (warp < 2 ? in && c0 < w : in && lane < n + 2) {
            unsigned o[3] = {row_at(yw - 1), row_at(yw), row_at(yw + 1)};
            V2<A> h[9];
            if (warp < 2) {
#pragma unroll
                for (int r = 0; r < 3; ++r) o[r] += xo;
                pull_rows<BC, A>(h, yw == 0, yw == ny - 1, [&](int a, int r, int dx) {
                    return pair_at<T>(plane_bytes(gin, plane, a), o[r], dx);
                });
            } else {
                int xa = x0 - 1, xb = x0 + w;
                if (BC == 2) {        // open sides: psi beyond is that of the edge column
                    if (x0 == 0) xa = 0;
                    if (xb == nx) xb = nx - 1;
                }
                const unsigned oa = (unsigned)xa * (unsigned)sizeof(T), ob = (unsigned)xb * (unsigned)sizeof(T);
                pull_rows<BC, A>(h, yw == 0, yw == ny - 1, [&](int a, int r, int dx) {
                    return two_at<T>(plane_bytes(gin, plane, a), o[r] + oa, o[r] + ob, dx);
                });
            }
            const V2<A> psi = eos_psi2<A, EOS, PLAIN_OF<T>>(site_rho<T>(h, P), P, warp == 2 || both, bad);
            A *ps = psis[yr - y0 + 1];
            if (warp == 2) {
                ps[1] = psi.lo();
                ps[w + 2] = psi.hi();
            } else if (both) {
                store_pair<A>(ps + c0 + 2, psi, true);
            } else {
                ps[c0 + 2] = psi.lo();
            }
        }
    }
    if (act) {
        const V2<A> psi = eos_psi2<A, EOS, PLAIN_OF<T>>(site_rho<T>(f, P), P, both, bad);
        A *ps = psis[warp + 1];
        if (both) store_pair<A>(ps + c0 + 2, psi, true);
        else ps[c0 + 2] = psi.lo();
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, ERR_DOMAIN);
    if (!act) return;

    finish_tile<T, BC, SR>(f, psis, P, gout, x0, x, y, warp, w, both, nx, ny, pitch, plane);
}

template <typename T, int EOS, int BC, int R, bool SR>
__global__ void __launch_bounds__(32 * R, tile_ctas(R, SR))
k_tile_step(const T *__restrict__ gin, T *__restrict__ gout,
            const __grid_constant__ DevConsts<Arith<T>> P, const int nx, const int ny,
            const int pitch, const unsigned plane, const int order, int *__restrict__ err) {
    __shared__ __align__(16) Arith<T> psis[R + 2][TILE_PW];
    // odd time steps visit the tiles in reverse: the rows the previous step wrote last, still
    // in L2, are read first
    const int bx = order ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
    const int by = order ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;
    tile_step<T, EOS, BC, R, SR>(gin, gout, P, nx, ny, pitch, plane, bx * TILE_W, by * R, psis, err);
}

// ---------------------------------------------------------------- staged tiles

// Shared memory of a staged tile: of each plane group the R + 2 rows that its psi rows (one more on
// either side) pull from, one TMA box per group; the psi rows; the barrier of the loads.
template <typename T, int R>
struct StagedSmem {
    static constexpr int ROWS = R + 2;
    static constexpr int GROUP = ((3 * ROWS * TILE_BOX_W * (int)sizeof(T) + 127) / 128) * 128 / (int)sizeof(T);
    __align__(128) T pop[3 * GROUP];
    __align__(16) Arith<T> psis[ROWS][TILE_PW];
    uint64_t bar;
};

// resident CTAs the staged kernels are compiled for: 64 registers per thread (128 with the
// stochastic-rounding hash)
__host__ __device__ constexpr int staged_ctas(int R, bool sr) {
    return 65536 / (32 * R * (sr ? 128 : 64));
}

// bytes that a staged tile expects and nobody sends: none but for the test hook (lb_debug_stall_row),
// which batches do not have
template <typename T>
__device__ __forceinline__ unsigned vain_bytes(const DevConsts<T> &P) { return P.vain_bytes; }
template <typename C>
__device__ __forceinline__ constexpr unsigned vain_bytes(const ConstFields<C> &) { return 0; }

// As tile_step, with the populations brought into shared memory by three TMA loads, so that a
// pull is a load at a constant offset: no address arithmetic, no wrap (414 instead of 471 warp
// instructions per 64 sites). The loads take longer to arrive than a warp's own, so the direct
// tile is ahead while latency counts; where memory is the bound, with walls and in BF16 this
// one is. Tiles whose rows wrap around a periodic lattice read global memory instead. Two
// variations were slower: the same with a persistent CTA that requests the next tile while it
// works on one (1024^2 14.2 against 12.2 us: 24 instead of 32 warps per SM, 493 instructions),
// and two rows per thread.
// CONSTS: P is being written to shared memory by the CTA (a barrier comes before its first use).
template <typename T, int EOS, int BC, int R, bool SR, bool CONSTS, typename PT>
__device__ __forceinline__ void staged_tile_step(const CUtensorMap *tmap,
                                                 const T *__restrict__ gin, T *__restrict__ gout,
                                                 const PT &P, const int nx, const int ny,
                                                 const int pitch, const unsigned plane, const int x0,
                                                 const int y0, StagedSmem<T, R> &sm,
                                                 int *__restrict__ err) {
    static_assert(R >= 3, "three warps carry the rim");
    using A = Arith<T>;
    using SM = StagedSmem<T, R>;
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int w = min(TILE_W, nx - x0), n = min(R, ny - y0);
    const int y = y0 + warp, c0 = 2 * lane, x = x0 + c0;
    const bool act = warp < n && c0 < w, both = c0 + 1 < w;
    const bool staged = tile_staged(BC, y0, R, ny);   // CTA-uniform

    if (staged && threadIdx.x == 0) {
        mbar_init(&sm.bar, 1);
        fence_mbar_init();
    }
    grid_dependency_wait();           // the previous step's state (programmatic dependent launch)
    grid_dependents_launch();
    if (staged && threadIdx.x == 0) {
        mbar_arrive_expect_tx(&sm.bar, 9u * SM::ROWS * TILE_BOX_W * (unsigned)sizeof(T) + vain_bytes(P));
#pragma unroll
        for (int q = 0; q < 3; ++q)   // rows outside the lattice (walls, open top) are zero-filled, not used
            tma_load_3d(sm.pop + q * SM::GROUP, tmap, x0 + GH<T> - TILE_BOX_LEFT, y0 - 2 + q, 3 * q, &sm.bar);
    }
    if (staged || CONSTS) __syncthreads();   // the barrier is initialised, the constants are written

    V2<A> f[9], h[9];
    // the rim: a row below or above the tile (warps 0, 1) or the two columns beside it (warp 2,
    // one row per lane)
    const int yr = warp == 0 ? y0 - 1 : warp == 1 ? y0 + n : y0 - 1 + lane;
    bool rim = warp < 2 ? c0 < w : warp == 2 && lane < n + 2;
    if (BC != 0) rim = rim && yr >= 0 && yr < ny;            // else psi is the edge row's
    int xa = x0 - 1, xb = x0 + w;     // open sides: psi beyond is that of the edge column
    if (BC == 2 && x0 == 0) xa = 0;
    if (BC == 2 && xb == nx) xb = nx - 1;

    if (staged) {
        if (!mbar_wait_bounded(&sm.bar, 0)) {     // give up: flag it, let the loads land, go on
            atomicOr(err, ERR_TIMEOUT);
            (void)mbar_wait_bounded(&sm.bar, 0);
        }
        // population a of lattice row yy + r - 1 at column xx + dx
        auto at = [&](int a, int r, int yy, int xx, int dx) -> const T * {
            const int q = plane_of(a) / 3, p = plane_of(a) % 3;
            return sm.pop + q * SM::GROUP + (p * SM::ROWS + (yy - y0) + r + 1 - q) * TILE_BOX_W +
                   (xx - x0) + TILE_BOX_LEFT + dx;
        };
        auto pair = [&](int a, int r, int yy, int dx) -> V2<A> {
            const T *s = at(a, r, yy, x, dx);
            if (dx == 0) return ring_pair<T>(s);
            return V2<A>(stored_val<T>(s[0]), stored_val<T>(s[1]));
        };
        if (act)
            pull_rows<BC, A>(f, y == 0, y == ny - 1, [&](int a, int r, int dx) { return pair(a, r, y, dx); });
        if (warp < 2) {
            if (rim)
                pull_rows<BC, A>(h, yr == 0, yr == ny - 1, [&](int a, int r, int dx) { return pair(a, r, yr, dx); });
        } else if (warp == 2) {
            if (rim)
                pull_rows<BC, A>(h, yr == 0, yr == ny - 1, [&](int a, int r, int dx) {
                    return V2<A>(stored_val<T>(*at(a, r, yr, xa, dx)), stored_val<T>(*at(a, r, yr, xb, dx)));
                });
        }
    } else {
        auto at = [&](int a, int r, int yy, int xx, int dx) -> const T * {
            int row = yy + r - 1;
            if (BC == 0) row = row < 0 ? row + ny : (row >= ny ? row - ny : row);
            return gin + (size_t)plane_of(a) * plane + (unsigned)row * (unsigned)pitch +
                   (unsigned)(xx + dx + GH<T>);
        };
        const int yw = BC == 0 ? (yr < 0 ? yr + ny : (yr >= ny ? yr - ny : yr)) : yr;
        if (act)
            pull_rows<BC, A>(f, y == 0, y == ny - 1, [&](int a, int r, int dx) {
                return V2<A>(stored_val<T>(*at(a, r, y, x, dx)), stored_val<T>(*at(a, r, y, x + 1, dx)));
            });
        if (warp != 2) {
            xa = x;
            xb = x + 1;
        }
        if (rim)
            pull_rows<BC, A>(h, yw == 0, yw == ny - 1, [&](int a, int r, int dx) {
                return V2<A>(stored_val<T>(*at(a, r, yw, xa, dx)), stored_val<T>(*at(a, r, yw, xb, dx)));
            });
    }

    bool bad = false;
    if (rim) {
        const V2<A> psi = eos_psi2<A, EOS, PLAIN_OF<T>>(site_rho<T>(h, P), P, warp == 2 || both, bad);
        A *ps = sm.psis[yr - y0 + 1];
        if (warp == 2) {
            ps[1] = psi.lo();
            ps[w + 2] = psi.hi();
        } else if (both) {
            store_pair<A>(ps + c0 + 2, psi, true);
        } else {
            ps[c0 + 2] = psi.lo();
        }
    }
    if (act) {
        const V2<A> psi = eos_psi2<A, EOS, PLAIN_OF<T>>(site_rho<T>(f, P), P, both, bad);
        A *ps = sm.psis[warp + 1];
        if (both) store_pair<A>(ps + c0 + 2, psi, true);
        else ps[c0 + 2] = psi.lo();
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, ERR_DOMAIN);
    if (!act) return;

    finish_tile<T, BC, SR>(f, sm.psis, P, gout, x0, x, y, warp, w, both, nx, ny, pitch, plane);
}

template <typename T, int EOS, int BC, int R, bool SR>
__global__ void __launch_bounds__(32 * R, staged_ctas(R, SR))
k_staged_tile_step(const __grid_constant__ CUtensorMap tin, const T *__restrict__ gin,
                   T *__restrict__ gout, const __grid_constant__ DevConsts<Arith<T>> P, const int nx,
                   const int ny, const int pitch, const unsigned plane, const int order,
                   int *__restrict__ err) {
    __shared__ StagedSmem<T, R> sm;
    const int bx = order ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
    const int by = order ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;
    staged_tile_step<T, EOS, BC, R, SR, false>(&tin, gin, gout, P, nx, ny, pitch, plane, bx * TILE_W,
                                               by * R, sm, err);
}

// Many periodic lattices: CTA (t, k) takes tile t of lattice k of the group. The lattice's
// constants go to shared memory as pairs, which the packed operations take as loaded, while the
// populations are on their way.
template <typename T, int EOS, int R>
__global__ void __launch_bounds__(32 * R, staged_ctas(R, false))
k_batch_tile(const __grid_constant__ BatchGroup G, const CUtensorMap *__restrict__ maps,
             const BatchLattice<T> *__restrict__ lats, const int phase, int *__restrict__ errs) {
    __shared__ StagedSmem<T, R> sm;
    __shared__ __align__(16) ConstFields<V2<T>> P;
    constexpr int NF = sizeof(ConstFields<T>) / sizeof(T);
    static_assert(sizeof(ConstFields<V2<T>>) == NF * sizeof(V2<T>) && NF <= 32 * R, "one field per thread");
    // phase 1 (every other step) visits the lattices and their tiles in reverse (see k_tile_step)
    const BatchGroup::Lattice &L = G.l[phase ? gridDim.y - 1 - blockIdx.y : blockIdx.y];
    const int t = phase ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
    const int x0 = t % L.tiles_x * TILE_W, y0 = t / L.tiles_x * R;
    if (y0 >= L.ny) return;           // a smaller lattice than the group's largest
    if (threadIdx.x < NF) {
        const T v = reinterpret_cast<const T *>(static_cast<const ConstFields<T> *>(&lats[L.lat].P))[threadIdx.x];
        reinterpret_cast<V2<T> *>(&P)[threadIdx.x] = V2<T>(v, v);
    }
    const T *gin = static_cast<const T *>(phase ? L.g[1] : L.g[0]);
    T *gout = static_cast<T *>(phase ? L.g[0] : L.g[1]);
    staged_tile_step<T, EOS, 0, R, false, true>(maps + 2 * L.lat + phase, gin, gout, P, L.nx, L.ny,
                                                L.pitch, L.plane, x0, y0, sm, &errs[L.lat]);
}

// ---------------------------------------------------------------- FP64: two passes

// FP64 is bound by GB300's FP64 pipe (2 operations per clock and SM), so nothing is computed
// twice: a psi pass stores psi (padded like a population plane, with the images of the edge
// columns beside it) and a collision pass reads it; the 16 extra bytes per site cost nothing
// beside the pipe. One site per thread: any lattice spreads over all SMs. Per step: 128^2 8.9
// against 118 us in the ring kernel (16 CTAs), 1000 x 700 219 against 280 us (which forms psi
// of the strip's rim in a pass of its own); 0.85 of the measured FP64 rate at 2048^2.
constexpr int SPLIT_THREADS = 64;

template <typename T, int BC>
__device__ __forceinline__ void pull_site(V1<T> (&f)[9], const T *__restrict__ g, unsigned plane,
                                          unsigned pitch, int x, int y, int ny) {
    int ym = y - 1, yp = y + 1;
    if (BC == 0) {
        ym = ym < 0 ? ny - 1 : ym;
        yp = yp >= ny ? 0 : yp;
    } else {
        ym = ym < 0 ? 0 : ym;
        yp = yp >= ny ? ny - 1 : yp;
    }
    const unsigned col = (unsigned)(x + GH<T>);
    const unsigned rm = (unsigned)ym * pitch + col, rz = (unsigned)y * pitch + col,
                   rp = (unsigned)yp * pitch + col;
    auto at = [&](int a, unsigned i) { return V1<T>(g[(size_t)plane_of(a) * plane + i]); };
    f[0] = at(0, rz);
    f[1] = at(1, rz - 1);
    f[3] = at(3, rz + 1);
    if (BC != 0 && y == 0) {
        f[2] = at(4, rz);
        f[5] = at(7, rz);
        f[6] = at(8, rz);
    } else {
        f[2] = at(2, rm);
        f[5] = at(5, rm - 1);
        f[6] = at(6, rm + 1);
    }
    if (BC == 1 && y == ny - 1) {
        f[4] = at(2, rz);
        f[7] = at(5, rz);
        f[8] = at(6, rz);
    } else {
        f[4] = at(4, rp);
        f[7] = at(7, rp + 1);
        f[8] = at(8, rp - 1);
    }
}

template <typename T, int EOS, int BC>
__global__ void __launch_bounds__(SPLIT_THREADS)
k_psi_site(const T *__restrict__ g, T *__restrict__ psi, const __grid_constant__ DevConsts<T> P,
           const int nx, const int ny, const int pitch, const unsigned plane,
           int *__restrict__ err) {
    const int x = blockIdx.x * SPLIT_THREADS + threadIdx.x, y = blockIdx.y;
    grid_dependency_wait();
    grid_dependents_launch();
    bool bad = false;
    if (x < nx) {
        V1<T> f[9];
        pull_site<T, BC>(f, g, plane, (unsigned)pitch, x, y, ny);
        const V1<T> rho = f[0] + (((f[1] + f[3]) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8])));
        const T v = eos_psi<T, EOS>(rho.v, P, bad);
        T *row = psi + (unsigned)y * (unsigned)pitch + GH<T>;
        row[x] = v;
        if (x == 0) row[BC == 2 ? -1 : nx] = v;           // images of the edge columns
        if (x == nx - 1) row[BC == 2 ? nx : -1] = v;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, ERR_DOMAIN);
}

template <typename T, int BC>
__global__ void __launch_bounds__(SPLIT_THREADS)
k_collide_site(const T *__restrict__ g, const T *__restrict__ psi, T *__restrict__ gout,
               const __grid_constant__ DevConsts<T> P, const int nx, const int ny,
               const int pitch, const unsigned plane) {
    const int x = blockIdx.x * SPLIT_THREADS + threadIdx.x, y = blockIdx.y;
    grid_dependency_wait();
    grid_dependents_launch();
    if (x >= nx) return;
    V1<T> f[9], pn[9];
    pull_site<T, BC>(f, g, plane, (unsigned)pitch, x, y, ny);
    int ym = y - 1, yp = y + 1;
    if (BC == 0) {
        ym = ym < 0 ? ny - 1 : ym;
        yp = yp >= ny ? 0 : yp;
    } else {                           // psi beyond a wall or the open top: the edge row's
        ym = ym < 0 ? 0 : ym;
        yp = yp >= ny ? ny - 1 : yp;
    }
    const T *pz = psi + (unsigned)y * (unsigned)pitch + GH<T> + x;
    const T *pm = psi + (unsigned)ym * (unsigned)pitch + GH<T> + x;
    const T *pp = psi + (unsigned)yp * (unsigned)pitch + GH<T> + x;
    pn[0] = pz[0]; pn[1] = pz[1]; pn[3] = pz[-1];
    pn[2] = pp[0]; pn[5] = pp[1]; pn[6] = pp[-1];
    pn[4] = pm[0]; pn[8] = pm[1]; pn[7] = pm[-1];
    collide<T, BC == 2>(f, pn, P);
    const unsigned rowi = (unsigned)y * (unsigned)pitch;
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        T *row = gout + (size_t)plane_of(a) * plane + rowi + GH<T>;
        row[x] = f[a].v;
        if (BC == 2) {
            if (x == 0) row[-1] = row[-2] = f[a].v;
            if (x == nx - 1) row[nx] = row[nx + 1] = f[a].v;
        } else {
            if (x < 2) row[nx + x] = f[a].v;
            if (x >= nx - 2) row[x - nx] = f[a].v;
        }
    }
}

// ---------------------------------------------------------------- dispatch

// launch with programmatic dependent launch (each kernel waits before its first access)
template <typename K, typename... Args>
cudaError_t launch_dependent(K kern, dim3 grid, dim3 block, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// a step's launch, or the kernel's resident CTAs per SM (StepBuffers::occ)
template <typename K, typename... Args>
cudaError_t launch_or_count(const StepBuffers &b, K kern, dim3 grid, dim3 block, cudaStream_t st, Args... args) {
    if (!b.occ) return launch_dependent(kern, grid, block, st, args...);
    int n = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, (int)block.x, 0);
    *b.occ = std::min(*b.occ, n);
    return e;
}

template <typename T, int EOS, int BC>
cudaError_t tile_launch(const Consts &c, const Geom &g, int variant, int order,
                        const StepBuffers &b, int *err, cudaStream_t st) {
    constexpr bool BF = std::is_same<T, __nv_bfloat16>::value;
    const int tx = (g.nx + TILE_W - 1) / TILE_W;
    const T *gin = static_cast<const T *>(b.gin);
    T *gout = static_cast<T *>(b.gout);
    if (variant == direct_variant()) {
        constexpr int R = DIRECT_ROWS;
        auto kern = k_tile_step<T, EOS, BC, R, false>;
        if constexpr (BF) {
            if (c.stochastic) kern = k_tile_step<T, EOS, BC, R, true>;
        }
        return launch_or_count(b, kern, dim3(tx, (g.ny + R - 1) / R), dim3(32 * R), st, gin, gout, to_dev<Arith<T>>(c),
                               g.nx, g.ny, g.pitch, (unsigned)g.plane, order, err);
    }
    constexpr int R = STAGED_ROWS;
    auto kern = k_staged_tile_step<T, EOS, BC, R, false>;
    if constexpr (BF) {
        if (c.stochastic) kern = k_staged_tile_step<T, EOS, BC, R, true>;
    }
    return launch_or_count(b, kern, dim3(tx, (g.ny + R - 1) / R), dim3(32 * R), st,
                           *static_cast<const CUtensorMap *>(b.tensor_map_in), gin, gout,
                           to_dev<Arith<T>>(c), g.nx, g.ny, g.pitch, (unsigned)g.plane, order, err);
}

template <typename T, int EOS>
cudaError_t tile_bc(const Consts &c, const Geom &g, int variant, int order,
                    const StepBuffers &b, int *err, cudaStream_t st) {
    switch (g.walls) {
        case 0: return tile_launch<T, EOS, 0>(c, g, variant, order, b, err, st);
        case 1: return tile_launch<T, EOS, 1>(c, g, variant, order, b, err, st);
        default:
            // open boundaries (and nu(rho)) are compiled for FP32 and FP64 only
            if constexpr (std::is_same<T, __nv_bfloat16>::value) return cudaErrorInvalidValue;
            else return tile_launch<T, EOS, 2>(c, g, variant, order, b, err, st);
    }
}

template <typename T>
cudaError_t tile_dispatch(const Consts &c, const Geom &g, int variant, int order,
                          const StepBuffers &b, int *err, cudaStream_t st) {
    switch (c.eos_kind) {
        case LB_EOS_CS: return tile_bc<T, LB_EOS_CS>(c, g, variant, order, b, err, st);
        case LB_EOS_EXP: return tile_bc<T, LB_EOS_EXP>(c, g, variant, order, b, err, st);
        default: return tile_bc<T, LB_EOS_PIECEWISE>(c, g, variant, order, b, err, st);
    }
}

template <typename T>
cudaError_t batch_tile_dispatch(int eos, const BatchGroup &group, int n, int max_tiles,
                                const void *maps, const void *lats, int phase, int *errs,
                                cudaStream_t st) {
    constexpr int R = STAGED_ROWS;
    auto kern = eos == LB_EOS_CS    ? k_batch_tile<T, LB_EOS_CS, R>
                : eos == LB_EOS_EXP ? k_batch_tile<T, LB_EOS_EXP, R>
                                    : k_batch_tile<T, LB_EOS_PIECEWISE, R>;
    return launch_dependent(kern, dim3(max_tiles, n), dim3(32 * R), st, group,
                            static_cast<const CUtensorMap *>(maps),
                            static_cast<const BatchLattice<T> *>(lats), phase, errs);
}

template <typename T, int EOS, int BC>
cudaError_t split_launch(const Consts &c, const Geom &g, const StepBuffers &b, int *err, cudaStream_t st) {
    const dim3 grid((g.nx + SPLIT_THREADS - 1) / SPLIT_THREADS, g.ny);
    const DevConsts<T> P = to_dev<T>(c);
    const T *gin = static_cast<const T *>(b.gin);
    T *psi = static_cast<T *>(b.psi), *gout = static_cast<T *>(b.gout);
    cudaError_t e = launch_or_count(b, k_psi_site<T, EOS, BC>, grid, dim3(SPLIT_THREADS), st, gin, psi, P, g.nx,
                                    g.ny, g.pitch, (unsigned)g.plane, err);
    if (e != cudaSuccess) return e;
    return launch_or_count(b, k_collide_site<T, BC>, grid, dim3(SPLIT_THREADS), st, gin, (const T *)psi, gout, P,
                           g.nx, g.ny, g.pitch, (unsigned)g.plane);
}

template <typename T, int EOS>
cudaError_t split_bc(const Consts &c, const Geom &g, const StepBuffers &b, int *err, cudaStream_t st) {
    switch (g.walls) {
        case 0: return split_launch<T, EOS, 0>(c, g, b, err, st);
        case 1: return split_launch<T, EOS, 1>(c, g, b, err, st);
        default: return split_launch<T, EOS, 2>(c, g, b, err, st);
    }
}

}  // namespace

}  // namespace lbm
