// Many time steps of a mid-size FP32 lattice in one launch: every SM keeps one tile of the lattice in
// shared memory (k_resident_steps). Same arithmetic and results, bit for bit, as the step kernels of
// lb_step.cuh and lb_tile.cuh.
#include <algorithm>

#include "lb_tile.cuh"

namespace lbm {

namespace {

constexpr int RS_W = TILE_W;          // columns of a tile (the last of a row may have fewer, at least 2)
constexpr int RS_STRIDE = 70;         // row stride: columns -2 .. 65, and lanes a row apart in 16 banks
constexpr int RS_MAX_ROWS = 35;       // rows of a tile that fit shared memory
constexpr int RS_BORDER = 8;          // warps of the border
constexpr int RS_INNER = 16;          // warps of the interior, at most
constexpr int RS_FETCH = 7;           // halo values a thread has in flight
constexpr int RS_ROW_SLOTS = 18, RS_COL_SLOTS = 36;

// storage plane p holds a population that moves in y by 1 - p / 3 and in x by plane_ex(p)
__host__ __device__ constexpr int plane_ex(int p) {
    for (int a = 0; a < 9; ++a)
        if (plane_of(a) == p) return EXv(a);
    return 0;
}
__host__ __device__ constexpr int plane_ey(int p) {
    for (int a = 0; a < 9; ++a)
        if (plane_of(a) == p) return EYv(a);
    return 0;
}
static_assert(plane_ey(0) == 1 && plane_ey(2) == 1 && plane_ey(3) == 0 && plane_ey(5) == 0 &&
                  plane_ey(6) == -1 && plane_ey(8) == -1,
              "plane groups are ordered by the row they are pulled from");

// How a lattice is cut: tx x ty tiles of RS_W columns and rows [ny k / ty, ny (k + 1) / ty).
struct ResidentShape {
    int tx, ty, max_rows, inner;      // inner: warps of the interior
};
__host__ __device__ constexpr int max_items(int rows) { return RS_ROW_SLOTS * (RS_W + 4) + RS_COL_SLOTS * rows; }

// The exchange words behind the epoch (word 0: steps taken by earlier launches; word 1: CTAs of this
// launch that are done): two copies (even and odd steps) of
//   rows:    [ty][18][64 tx]  of a tile's row 0 planes 3..8, row 1 planes 6..8, last row planes 0..5,
//                             last but one planes 0..2
//   columns: [tx][4][9][ny]   of its column 0, column 1, last, last but one
//   one that nobody publishes (the test hook, see lb_debug_stall_row, waits for it)
// A word is a value and the time (epoch + step) it belongs to.
__host__ __device__ constexpr unsigned row_words(int tx, int ty) { return (unsigned)ty * RS_ROW_SLOTS * RS_W * (unsigned)tx; }
__host__ __device__ constexpr unsigned col_words(int tx, int ny) { return (unsigned)tx * RS_COL_SLOTS * (unsigned)ny; }
__host__ __device__ constexpr unsigned exchange_words(int tx, int ty, int ny) {
    return row_words(tx, ty) + col_words(tx, ny) + 4;   // (a sector: the copies stay aligned)
}

__device__ __forceinline__ uint64_t load_word(const uint64_t *p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void store_word(uint64_t *p, float v, unsigned tag) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p),
                 "l"(((uint64_t)tag << 32) | __float_as_uint(v)) : "memory");
}

// named barriers among `threads` threads of the CTA: wait for them, or be counted only
__device__ __forceinline__ void bar_wait(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// n_steps time steps of one lattice, two at least. gout may be gin: a tile stores its last step when its
// neighbours have published their first, after they have read the state. The tile's populations lie in two copies in shared memory
// (even and odd steps), [9][rows + 4][70]: its sites and two halo cells on every side. Eight warps
// take the border (the outer two rows and pairs of columns) and the halo: fetch it, psi of the
// outermost rows and columns and of the ones around the tile, collide, publish. The others take what
// needs no halo meanwhile: psi, then the collision of the interior.
// A published value carries its time in the same 64-bit word, so that the reader polls the value
// itself: no fence, no flag, one trip through L2. Two copies of the exchange words suffice: a tile
// publishes time t + 2 after it has read its neighbours' t + 1, which they publish after they have
// read t. All CTAs must be resident (cooperative launch); a wait gives up after a second, once per
// CTA, and the launch then ends with ERR_TIMEOUT.
// What bounds it: the border's chain, in clocks of 501 x 383 (64 x 20 tiles): 2500 until the halo is
// here, 1000 psi, 2100 collision and publishing, with the interior beside it; 2.3 us a step at
// least. Per step, against a launch of the tile kernels per step: 256^2 2.3 / 2.7 us, 384^2 2.8 / 3.3,
// 501 x 383 3.1 / 4.5, 512^2 3.7 / 4.4, 560^2 4.2 / 5.1, 600 x 225 splash 3.4 / 3.9. The same warps
// for border and interior took 4.1 us at 501 x 383; polling one value after the other 3.7.
template <int EOS, int BC>
__global__ void __launch_bounds__(32 * (RS_BORDER + RS_INNER), 1)
k_resident_steps(const float *gin, float *gout,
                 const __grid_constant__ DevConsts<float> P, const int nx, const int ny,
                 const int pitch, const unsigned plane, const int n_steps, const int ty,
                 const int max_rows, uint64_t *__restrict__ words, int *__restrict__ err) {
    extern __shared__ __align__(16) float rs_smem[];
    using T = float;
    __shared__ int dead_flag, n_items;
    volatile int *dead = &dead_flag;
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int warps = blockDim.x >> 5, inner = warps - RS_BORDER;
    const int tx = (nx + RS_W - 1) / RS_W, bx = (int)blockIdx.x % tx, by = (int)blockIdx.x / tx;
    const int x0 = bx * RS_W, w = min(RS_W, nx - x0);
    const int y0 = ny * by / ty, n = ny * (by + 1) / ty - y0;
    const int PS = (max_rows + 4) * RS_STRIDE;
    float *const psis = rs_smem + 18 * PS;                    // rows -1 .. n
    int2 *const items = reinterpret_cast<int2 *>(psis + (max_rows + 2) * RS_STRIDE);
    const unsigned n_words = exchange_words(tx, ty, ny);
    uint64_t *const exch = words + 2;
    const unsigned epoch = (unsigned)load_word(words);
    const int c0 = 2 * lane, cr = (w - 1) & ~1;               // the lane's pair, the last pair
    if (threadIdx.x == 0) dead_flag = 0, n_items = 0;
    __syncthreads();

    // what arrives each step: (exchange word, place in shared memory) per halo value
    const int wide = w + 4, row_items = RS_ROW_SLOTS * wide;
    for (int base = 32 * warp; base < row_items + RS_COL_SLOTS * n; base += (int)blockDim.x) {
        const int i = base + lane;
        int2 it = make_int2(-1, 0);
        int from = 0;                             // the lattice row it comes from
        if (i < row_items) {
            // slots as published: the row above the tile is row 0 or 1 of the next tile
            const int slot = i / wide, col = i - slot * wide - 2;
            const int row = slot < 6 ? n : slot < 9 ? n + 1 : slot < 15 ? -1 : -2;
            const int p = slot < 6 ? slot + 3 : slot < 9 ? slot : slot < 15 ? slot - 9 : slot - 15;
            int nb = slot < 9 ? by + 1 : by - 1, gx = x0 + col;
            const bool in = BC == 0 || (nb >= 0 && nb < ty);
            nb = nb < 0 ? ty - 1 : nb >= ty ? 0 : nb;
            from = y0 + row < 0 ? y0 + row + ny : y0 + row >= ny ? y0 + row - ny : y0 + row;
            if (BC == 2) gx = gx < 0 ? 0 : gx >= nx ? nx - 1 : gx;
            else gx = gx < 0 ? gx + nx : gx >= nx ? gx - nx : gx;
            if (in)
                it = make_int2((nb * RS_ROW_SLOTS + slot) * RS_W * tx + gx, p * PS + (row + 2) * RS_STRIDE + col + 2);
        } else if (i < row_items + RS_COL_SLOTS * n) {
            const int slot = (i - row_items) / n, r = i - row_items - slot * n;
            const int s = slot / 9, p = slot - 9 * s;
            int nb = s < 2 ? bx + 1 : bx - 1;
            const int col = s == 0 ? w : s == 1 ? w + 1 : s == 2 ? -1 : -2;
            // beside open sides the tile's own threads copy the edge column; of the inner halo column
            // the populations that leave the tile are not pulled (but beside a wall, whose bounced
            // links read their own site), of the outer one only those that enter it
            bool in = BC != 2 || (nb >= 0 && nb < tx);
            const int ex = plane_ex(p), into = s < 2 ? -1 : 1;
            if (BC == 0) in = in && ((s & 1) ? ex == into : ex != -into);
            nb = nb < 0 ? tx - 1 : nb >= tx ? 0 : nb;
            from = y0 + r;
            if (in)
                it = make_int2((int)row_words(tx, ty) + (nb * RS_COL_SLOTS + slot) * ny + y0 + r,
                               p * PS + (r + 2) * RS_STRIDE + col + 2);
        }
        if (it.x >= 0 && from == P.stall_row) it.x = (int)n_words - 1;   // test hook
        const unsigned have = __ballot_sync(0xffffffffu, it.x >= 0);
        int at = 0;
        if (lane == 0) at = atomicAdd(&n_items, __popc(have));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(have & ((1u << lane) - 1u));
        if (it.x >= 0) items[at] = it;
    }

    // the state, two halo cells on every side (rows beyond a wall or the open top are not read)
    for (int j = warp; j < 9 * (n + 4); j += warps) {
        const int p = j / (n + 4), r = j - p * (n + 4);
        int y = y0 + r - 2;
        if (BC == 0) y = y < 0 ? y + ny : y >= ny ? y - ny : y;
        if (y < 0 || y >= ny) continue;
        const float *src = gin + (size_t)p * plane + (unsigned)y * (unsigned)pitch + (unsigned)(x0 + GH<T> - 2);
        for (int c = lane; c < wide; c += 32) rs_smem[p * PS + r * RS_STRIDE + c] = src[c];
    }
    __syncthreads();

    bool bad = false;
    const int count = n_items, m = n - 4;         // halo values; interior rows

    // The border's work in units of a warp, the lane's pair (r, c) of unit k; false: none.
    // psi: rows 0, n - 1, -1 and n, then the edge columns (then the columns beside the tile)
    const int edge = (2 * (n - 2) + 31) / 32, rim = (n + 2 + 31) / 32;
    auto psi_unit = [&](int k, int &r, int &c) {
        r = k == 0 ? 0 : k == 1 ? n - 1 : k == 2 ? -1 : n;
        c = c0;
        bool on = c < w;
        if (k >= 4) {
            const int i = (k - 4) * 32 + lane;
            r = 1 + (i >= n - 2 ? i - (n - 2) : i);
            c = i >= n - 2 ? cr : 0;
            on = i < 2 * (n - 2) && (i < n - 2 || cr > 0);
        }
        return on && (BC == 0 || (y0 + r >= 0 && y0 + r < ny));
    };
    // collisions: the outer two rows, then two pairs on either side of the rows between
    constexpr int brows = 4;
    const int bcols = (4 * m + 31) / 32;
    auto collide_unit = [&](int k, int &r, int &c) {
        r = k < 2 ? k : m + k;
        c = c0;
        if (k < brows) return c < w;
        const int i = (k - brows) * 32 + lane, side = (i >= m) + (i >= 2 * m) + (i >= 3 * m);
        r = 2 + i - side * m;
        c = side == 0 ? 0 : side == 1 ? cr : side == 2 ? 2 : cr - 2;
        return i < 4 * m && (side == 0 || (side == 1 ? cr >= 2 : side == 2 ? cr >= 4 : cr >= 6));
    };
    int pr, pc, qr, qc;                           // of the warp's first unit, for all steps
    const bool p_on = psi_unit(warp, pr, pc), q_on = collide_unit(warp, qr, qc);
#pragma unroll 1
    for (int t = 0; t < n_steps; ++t) {
        float *const S = rs_smem + (t & 1) * 9 * PS, *const N = rs_smem + ((t & 1) ^ 1) * 9 * PS;
        auto pull = [&](V2<T>(&f)[9], int r, int c) {
            const int y = y0 + r;
            const T *s0 = S + (r + 1) * RS_STRIDE + c + 2;
            pull_rows<BC, T>(f, y == 0, y == ny - 1, [&](int a, int row, int dx) {
                const T *s = s0 + plane_of(a) * PS + row * RS_STRIDE + dx;
                return dx == 0 ? lds_pair<T>(s) : V2<T>(s[0], s[1]);
            });
        };
        auto psi_pair = [&](int r, int c) {
            V2<T> f[9];
            pull(f, r, c);
            const V2<T> psi = eos_psi2<T, EOS>(rho_pair(f), P, c + 1 < w, bad);
            T *d = psis + (r + 1) * RS_STRIDE + c + 2;
            if (c + 1 < w) store_pair<T>(d, psi, true);
            else d[0] = psi.lo();
        };
        // collide the pair and store it: f as stored
        auto collide_pair = [&](V2<T>(&f)[9], int r, int c, bool both) {
            const int y = y0 + r;
            V2<T> pn[9];
            pull(f, r, c);
            const T *p0 = psis + (r + 1) * RS_STRIDE + c + 2;
            const T *pm = BC != 0 && y == 0 ? p0 : p0 - RS_STRIDE;
            const T *pp = BC != 0 && y == ny - 1 ? p0 : p0 + RS_STRIDE;
            const V2<T> m0 = lds_pair<T>(pm), z0 = lds_pair<T>(p0), q0 = lds_pair<T>(pp);
            pn[0] = z0;
            pn[1] = V2<T>(z0.hi(), p0[2]);
            pn[2] = q0;
            pn[3] = V2<T>(p0[-1], z0.lo());
            pn[4] = m0;
            pn[5] = V2<T>(q0.hi(), pp[2]);
            pn[6] = V2<T>(pp[-1], q0.lo());
            pn[7] = V2<T>(pm[-1], m0.lo());
            pn[8] = V2<T>(m0.hi(), pm[2]);
            collide<T, BC == 2>(f, pn, P);
            if (t + 1 == n_steps) {
                const int x = x0 + c;
                const unsigned rowi = (unsigned)y * (unsigned)pitch;
#pragma unroll
                for (int a = 0; a < 9; ++a)
                    store_pop_pair<T, false>(gout + (size_t)plane_of(a) * plane + rowi + (unsigned)(x + GH<T>), f[a], both, 0u);
                return;
            }
            T *d = N + (r + 2) * RS_STRIDE + c + 2;
#pragma unroll
            for (int a = 0; a < 9; ++a) {
                T *da = d + plane_of(a) * PS;
                if (both) store_pair<T>(da, f[a], true);
                else da[0] = f[a].lo();
            }
        };

        if (warp >= RS_BORDER) {
            for (int r = 1 + warp - RS_BORDER; r < n - 1; r += inner)
                if (c0 >= 2 && c0 + 2 < w) psi_pair(r, c0);
            bar_arrive(1, (int)blockDim.x);
            bar_wait(2, 32 * inner);                  // psi of the interior
            for (int r = 2 + warp - RS_BORDER; r < n - 2; r += inner)
                if (c0 >= 4 && c0 + 4 < w) {
                    V2<T> f[9];
                    collide_pair(f, r, c0, true);
                }
        } else {
            if (t > 0) {
                const uint64_t *src = exch + ((t & 1) ? n_words : 0u);
                const unsigned tag = epoch + (unsigned)t;
                for (int base = (int)threadIdx.x; base < count; base += RS_FETCH * 32 * RS_BORDER) {
                    // all of them at once, and again those whose time has not come
                    uint64_t v[RS_FETCH];
                    const uint64_t *from[RS_FETCH];
                    bool ready = true;
#pragma unroll
                    for (int k = 0; k < RS_FETCH; ++k) {
                        const int i = base + k * 32 * RS_BORDER;
                        v[k] = (uint64_t)tag << 32;
                        from[k] = src + (i < count ? items[i].x : 0);
                        if (i < count) v[k] = load_word(from[k]);
                    }
#pragma unroll
                    for (int k = 0; k < RS_FETCH; ++k) ready &= (unsigned)(v[k] >> 32) == tag;
                    if (!ready && !*dead) {
                        const uint64_t start = global_ns();
                        for (int tries = 0; !ready; ++tries) {
                            if ((tries & 63) == 63 && (*dead || global_ns() - start > 1000000000ull)) {
                                *dead = 1;                 // give up, and wait for nothing any more
                                atomicOr(err, ERR_TIMEOUT);
                                break;
                            }
#pragma unroll
                            for (int k = 0; k < RS_FETCH; ++k)
                                if ((unsigned)(v[k] >> 32) != tag) v[k] = load_word(from[k]);
                            ready = true;
#pragma unroll
                            for (int k = 0; k < RS_FETCH; ++k) ready &= (unsigned)(v[k] >> 32) == tag;
                        }
                    }
#pragma unroll
                    for (int k = 0; k < RS_FETCH; ++k) {
                        const int i = base + k * 32 * RS_BORDER;
                        if (i < count) S[items[i].y] = __uint_as_float((unsigned)v[k]);
                    }
                }
            }
            bar_wait(3, 32 * RS_BORDER);              // the halo is here
            // psi of the tile's edge rows and columns, and of the rows and columns around it
            for (int k = warp; k < 4 + edge + rim; k += RS_BORDER) {
                if (k < 4 + edge) {
                    int r = pr, c = pc;
                    const bool on = k == warp ? p_on : psi_unit(k, r, c);
                    if (on) psi_pair(r, c);
                } else {
                    const int r = (k - 4 - edge) * 32 + lane - 1, y = y0 + r;
                    if (r <= n && (BC == 0 || (y >= 0 && y < ny))) {
                        // open sides: psi beyond is that of the edge column
                        const int ca = BC == 2 && x0 == 0 ? 0 : -1, cb = BC == 2 && x0 + w == nx ? w - 1 : w;
                        V2<T> f[9];
                        pull_rows<BC, T>(f, y == 0, y == ny - 1, [&](int a, int row, int dx) {
                            const T *s = S + plane_of(a) * PS + (r + 1 + row) * RS_STRIDE + 2 + dx;
                            return V2<T>(s[ca], s[cb]);
                        });
                        const V2<T> psi = eos_psi2<T, EOS>(rho_pair(f), P, true, bad);
                        T *d = psis + (r + 1) * RS_STRIDE + 2;
                        d[-1] = psi.lo();
                        d[w] = psi.hi();
                    }
                }
            }
            bar_wait(1, (int)blockDim.x);             // all of psi

            const unsigned tag = epoch + (unsigned)t + 1u;
            uint64_t *const dst = exch + ((t & 1) ? 0u : n_words);
            for (int k = warp; k < brows + bcols; k += RS_BORDER) {
                int r = qr, c = qc;
                const bool on = k == warp ? q_on : collide_unit(k, r, c);
                if (!on) continue;
                const bool both = c + 1 < w;
                V2<T> f[9];
                collide_pair(f, r, c, both);
                if (t + 1 == n_steps) {
                    store_ghosts<T, BC, false>(gout, f, x0 + c, (unsigned)(y0 + r) * (unsigned)pitch, nx, plane, both, 0u);
                    continue;
                }
                if (BC == 2 && x0 == 0 && c == 0) {
#pragma unroll
                    for (int a = 0; a < 9; ++a) {
                        T *g = N + plane_of(a) * PS + (r + 2) * RS_STRIDE;
                        g[0] = g[1] = f[a].lo();
                    }
                }
                if (BC == 2 && x0 + w == nx && c == cr) {
#pragma unroll
                    for (int a = 0; a < 9; ++a) {
                        T *g = N + plane_of(a) * PS + (r + 2) * RS_STRIDE + w + 2;
                        g[0] = g[1] = both ? f[a].hi() : f[a].lo();
                    }
                }
                // planes p .. q - 1 of a row, to the slots from `slot`
                auto row_out = [&](int slot, int p, int q) {
                    uint64_t *d = dst + ((unsigned)(by * RS_ROW_SLOTS + slot) * RS_W * tx + (unsigned)(x0 + c));
#pragma unroll
                    for (int a = 0; a < 9; ++a) {
                        if (plane_of(a) < p || plane_of(a) >= q) continue;
                        uint64_t *e = d + (unsigned)(plane_of(a) - p) * (unsigned)(RS_W * tx);
                        store_word(e, f[a].lo(), tag);
                        if (both) store_word(e + 1, f[a].hi(), tag);
                    }
                };
                if (k < brows) {
                    if (r == 0) row_out(0, 3, 9);
                    if (r == 1) row_out(6, 6, 9);
                    if (r == n - 1) row_out(9, 0, 6);
                    if (r == n - 2) row_out(15, 0, 3);
                }
                auto col_out = [&](int s, bool hi) {
                    uint64_t *q = dst + (row_words(tx, ty) + (unsigned)(bx * RS_COL_SLOTS + 9 * s) * ny + (unsigned)(y0 + r));
#pragma unroll
                    for (int a = 0; a < 9; ++a) {
                        const int ex = EXv(a), out = s < 2 ? -1 : 1;
                        if (BC != 0 || ((s & 1) ? ex == out : ex != -out))
                            store_word(q + (unsigned)plane_of(a) * ny, hi ? f[a].hi() : f[a].lo(), tag);
                    }
                };
                if (c == 0) {
                    col_out(0, false);
                    col_out(1, true);                 // (w >= 2)
                }
                if (c == cr) {
                    col_out(2, both);
                    if (both) col_out(3, false);
                } else if (c + 3 == w) {
                    col_out(3, true);
                }
            }
        }
        __syncthreads();
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, ERR_DOMAIN);
    // every CTA has read the epoch: the last one moves it on for the next launch
    if (threadIdx.x == 0) {
        unsigned *done = reinterpret_cast<unsigned *>(words + 1);
        __threadfence();
        if (atomicAdd(done, 1u) == gridDim.x - 1) {
            *done = 0u;
            *words = (uint64_t)(epoch + (unsigned)n_steps);
        }
    }
}

constexpr int smem_of_rows(int rows) {
    return (18 * (rows + 4) + rows + 2) * RS_STRIDE * (int)sizeof(float) + max_items(rows) * (int)sizeof(int2);
}
int resident_smem(const ResidentShape &s) { return smem_of_rows(s.max_rows); }
constexpr int RS_SMEM_MOST = smem_of_rows(RS_MAX_ROWS);
static_assert(RS_SMEM_MOST + 1024 <= 228 * 1024, "a tile fits an SM (1 KB per CTA is the system's)");

// Tiles of at least 6 rows (with fewer there are more CTAs to exchange with and no less to wait for:
// 160^2 in tiles of 2, 4, 6, 12 rows 2.61, 2.30, 2.28, 2.62 us a step). false: the lattice does not fit,
// or steps by single launches are as fast, resident / single us a step: 176^2 2.29 / 2.15, 192^2 2.28 /
// 2.41, 256^2 2.30 / 2.70, 70 x 300 2.26 / 2.20, 400 x 100 2.27 / 2.41, 5000 x 20 (79 tiles) 3.11 / 2.72.
bool resident_shape(const Geom &g, int num_sms, ResidentShape &s) {
    s.tx = (g.nx + RS_W - 1) / RS_W;
    if (g.ny < 4 || g.nx < 4 || g.nx - (s.tx - 1) * RS_W < 2 || s.tx > num_sms) return false;
    s.ty = std::max(std::min(num_sms / s.tx, g.ny / 6), 1);
    if ((long long)g.nx * g.ny < 32768 || s.tx * s.ty < 96) return false;
    s.max_rows = (g.ny + s.ty - 1) / s.ty;
    if (s.max_rows > RS_MAX_ROWS) return false;
    // a warp for every interior row, every second or third
    const int rows = std::max(s.max_rows - 2, 1), passes = (rows + RS_INNER - 1) / RS_INNER;
    s.inner = (rows + passes - 1) / passes;
    return true;
}

template <int EOS, int BC>
cudaError_t resident_launch(const Consts &c, const Geom &g, const ResidentShape &s, const void *gin,
                            void *gout, int n_steps, uint64_t *words, int *err, cudaStream_t st, bool probe) {
    auto kern = k_resident_steps<EOS, BC>;
    const int smem = resident_smem(s);
    // the kernel's limit, not this lattice's size: contexts of several threads share the attribute
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, RS_SMEM_MOST);
    if (e != cudaSuccess) return e;
    if (probe) {
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, 32 * (RS_BORDER + s.inner), smem);
        return e != cudaSuccess ? e : n > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(s.tx * s.ty);
    cfg.blockDim = dim3(32 * (RS_BORDER + s.inner));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<const float *>(gin), static_cast<float *>(gout), to_dev<float>(c),
                              g.nx, g.ny, g.pitch, (unsigned)g.plane, n_steps, s.ty, s.max_rows, words, err);
}

template <int EOS>
cudaError_t resident_bc(const Consts &c, const Geom &g, const ResidentShape &s, const void *gin, void *gout,
                        int n_steps, uint64_t *words, int *err, cudaStream_t st, bool probe) {
    switch (g.walls) {
        case 0: return resident_launch<EOS, 0>(c, g, s, gin, gout, n_steps, words, err, st, probe);
        case 1: return resident_launch<EOS, 1>(c, g, s, gin, gout, n_steps, words, err, st, probe);
        default: return resident_launch<EOS, 2>(c, g, s, gin, gout, n_steps, words, err, st, probe);
    }
}

cudaError_t resident_dispatch(const Consts &c, const Geom &g, const ResidentShape &s, const void *gin, void *gout,
                              int n_steps, uint64_t *words, int *err, cudaStream_t st, bool probe) {
    switch (c.eos_kind) {
        case LB_EOS_CS: return resident_bc<LB_EOS_CS>(c, g, s, gin, gout, n_steps, words, err, st, probe);
        case LB_EOS_EXP: return resident_bc<LB_EOS_EXP>(c, g, s, gin, gout, n_steps, words, err, st, probe);
        default: return resident_bc<LB_EOS_PIECEWISE>(c, g, s, gin, gout, n_steps, words, err, st, probe);
    }
}

}  // namespace

// bytes of the exchange words (zero before the first launch), 0 if the lattice does not fit
size_t resident_bytes(int prec, const Consts &c, const Geom &g, int num_sms) {
    ResidentShape s;
    int dev = 0, coop = 0;
    if (prec != LB_FP32 || !resident_shape(g, num_sms, s)) return 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
        resident_dispatch(c, g, s, nullptr, nullptr, 0, nullptr, nullptr, nullptr, true) == cudaSuccess)
        return (2 + 2 * (size_t)exchange_words(s.tx, s.ty, g.ny)) * sizeof(uint64_t);
    (void)cudaGetLastError();
    return 0;
}

// every row is beside a tile of the next column of tiles, if there is one (around the lattice unless
// its sides are open)
bool resident_waits_for_row(const Geom &g, int row) {
    return row >= 0 && row < g.ny && (g.walls != 2 || g.nx > RS_W);
}

cudaError_t launch_resident_steps(const Consts &c, const Geom &g, int num_sms, const void *gin, void *gout,
                                  int n_steps, void *words, int *err, cudaStream_t st) {
    ResidentShape s;
    if (!resident_shape(g, num_sms, s)) return cudaErrorInvalidValue;
    return resident_dispatch(c, g, s, gin, gout, n_steps, static_cast<uint64_t *>(words), err, st, false);
}

}  // namespace lbm
