// lks_step_rows.cu -- kRowSteps steps of one lattice per pass over memory (FP32 and 16-bit storage).
//
// A single FP32 step moves 152 bytes a node and runs at the HBM rate, so more steps per second need
// fewer bytes per step: a block takes a strip of columns and marches up its rows, computing
// level 1 (the first step) of row r from global memory, level 2 of row r - 1 from the level-1
// rows it has just made, and so on; only the last level is stored.  Every level is the ordinary
// step (pull, wall closures, collision, rounding to the storage type), so the state after kRowSteps
// steps has the bits of as many single steps (but for the sign of a zero: without a body force the source terms,
// + 0, are left out, so a population of -0 may stay one).
//
// What the next level pulls from a level: populations with e_x = 0 come from the thread's own
// column and stay in registers (as storage words: the row above needs none of them back, the
// own row one, the row below two rows' worth); the ten with e_x != 0 pass through shared memory,
// in rings of three rows.  One block barrier per level and row orders them: a slot is written again
// two barriers after its last read.
//
// A strip carries kRowSteps - 1 extra columns on each side, and a chunk of rows as many extra rows
// at each end, recomputed by the neighbouring block; a row that fits one block wraps around
// instead.
//
// In place (one population buffer) a block overwrites rows and columns that its neighbours still have to
// pull from.  A copy kernel therefore saves kRowSteps rows or columns on either side of every block
// boundary first, and pulls that leave the block's own area read the copies.  Inside the area a row is
// stored two rows after its last pull.  The pass leaves the natural layout, as a pair of AA steps does.  The copies
// live in a workspace that the caller lends (lks_set_workspace).  FP32 in place, GLUPS, AA pairs -> fused with a body
// force / without one: 4096^2 45.2 -> 69.0 / 74.9, 2056 x 1500 43.3 -> 55.4 / 59.0, 2056 x 900 42.6 -> 47.7 / 51.0 (two
// buffers, fused: 4096^2 97.8 / 100.8, 2056 x 1500 96.1 / 102.5): the copies take 7 %, and the warp with the block's
// edges holds up the others at the barriers.
#include <algorithm>
#include <type_traits>

#include "lks_device.cuh"
#include "lks_internal.h"
#include "lks_packed.cuh"
#include "lks_pair.cuh"

namespace lks {
namespace {

// Rows of the first and last chunk, whose blocks test every row for a wall and run about 1.5 times as
// long a row, as a share of the others'.
constexpr double kEdgeShare = 0.65;
// Fewest rows of a chunk.  A pass costs about the same per row and block whatever the fit, kRowSteps - 1 rows more
// per chunk than it stores, so its rate is the share of the computed nodes that are the lattice's own (the plan's
// use) times 95-129 GLUPS for FP32, 107-133 for BF16, 105-115 for FP16 (measured over widths of 70 to 2048 and
// chunks of 4 to 106 rows).  Single steps: 43-57 (FP32), 45-73 (16-bit) while both buffers fit in L2, 39-45 and 44-57
// from memory.  GLUPS, fused against single: FP32 1000 x 513 (use 0.59) 53.6 / 57.4, 132 x 2800 (0.38) 39.7 / 50.3,
// 264 x 4000 (0.60, from memory) 67.7 / 41.1, 132 x 40000 (0.50, from memory) 64.7 / 40.3; FP16 1500 x 700 (0.61)
// 64.6 / 68.5, 900 x 1100 (0.64) 70.6 / 64.1, 264 x 2500 (0.39) 42.0 / 48.2; BF16 520 x 1500 (0.50) 59.4 / 59.2.
constexpr int kRowMinChunk = 8;
constexpr double kUseL2 = 0.62, kUseMemory = 0.47;
// In place the saved edges and the blocks' far pulls cost more, the AA pairs less: 1000^2 (0.73, in L2) 35 against 60,
// 2000 x 800 (0.78) 43.6 / 43.1, 2056 x 1500 (0.88) 55.7 / 43.1, 4096^2 68.4 / 45.0; 250 x 3000 (0.55, in L2) 23 / 54.
constexpr double kUseInPlace = 0.8;
// Rows fetched into L2 ahead of their first use (no prefetch: FP16 92.8 instead of 100.3 GLUPS).
constexpr int kAhead = 2;

// One node per thread: a word is a stored population.
template <typename S>
struct OneNode {
    typedef S W;
    typedef float V;
    static constexpr int kNodes = 1;
    static __device__ __forceinline__ V unpack(W w) { return Loader<S, float, false>::ld(&w); }
    static __device__ __forceinline__ W pack(V v) {
        W w;
        store_s<S, float>(&w, v);
        return w;
    }
    // the population pulled from x - 1 (x + 1), given the words of the left (right) and own columns
    static __device__ __forceinline__ W from_left(W left, W) { return left; }
    static __device__ __forceinline__ W from_right(W, W right) { return right; }
    static constexpr bool kOwn = false;  // own word unused by the two above
};

// Two x-adjacent nodes per thread (16-bit storage): a word holds both.
template <typename S>
struct TwoNodes {
    typedef uint32_t W;
    typedef float2 V;
    static constexpr int kNodes = 2;
    static __device__ __forceinline__ V unpack(W w) { return Packed<S>::pair(w); }
    static __device__ __forceinline__ W pack(V v) { return Packed<S>::pack(v.x, v.y); }
    static __device__ __forceinline__ W from_left(W left, W own) { return __byte_perm(left, own, 0x5432); }
    static __device__ __forceinline__ W from_right(W own, W right) { return __byte_perm(own, right, 0x5432); }
    static constexpr bool kOwn = true;
};

// FP16 words hold deviations times kHalfScale.  With the Maxwell coupling the two-node kernel leaves them
// scaled: the parameters that produce populations are scaled once on the host (scaled_params), and only
// the five moments are brought back.  A power of two commutes with every rounding here, so the bits are
// those of the unscaled form, for 5 multiplications a pair instead of 38 (FP16 107 -> 117 GLUPS at 4096^2).
template <typename S>
struct TwoNodesScaled : TwoNodes<S> {
    typedef uint32_t W;
    typedef float2 V;
    static __device__ __forceinline__ V unpack(W w) { return __half22float2(*reinterpret_cast<const __half2*>(&w)); }
    static __device__ __forceinline__ W pack(V v) {
        const __half2 h = __floats2half2_rn(v.x, v.y);
        return *reinterpret_cast<const uint32_t*>(&h);
    }
};
template <typename N> struct IsScaled { static constexpr bool value = false; };
template <typename S> struct IsScaled<TwoNodesScaled<S>> { static constexpr bool value = true; };

// Parameters of the scaled form: everything a population is made of that is not another population.
// The moment closure runs unscaled and keeps its kx.
StepParams<float> scaled_params(StepParams<float> p, int closure) {
    for (float* v : {&p.owf0, &p.owf1, &p.owf5, &p.owm0, &p.owm1, &p.sw0, &p.sw1, &p.sw5, &p.bot.du, &p.top.du})
        *v *= kHalfScale;
    if (closure == 0) p.bot.kx *= kHalfScale, p.top.kx *= kHalfScale;
    return p;
}

// collide_node and collide_g, the same operations in the same order, with two things it leaves to its caller:
// SCALED populations with scaled_params, whose moments are brought back here, and no body force (FORCE false:
// the source terms are zeros then, a sixth of the arithmetic; 4096^2 without a force, GLUPS: BF16 125 -> 141,
// FP16 117 -> 132, FP32, near the HBM rate, 97.8 -> 100.5).
template <bool FORCE, bool SCALED, typename V>
__device__ __forceinline__ void collide_rows(V f[9], V gx[5], V gy[5], const StepParams<float>& p) {
    const float half = 0.5f, three = 3.0f, four5 = 4.5f, one5 = 1.5f;
    auto back = [&](V x) -> V {
        if constexpr (SCALED) return fmul(kHalfUnscale, x);
        return x;
    };
    const auto drho = back(((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8]);
    const auto rho = 1.0f + drho;
    const auto jx = back((f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]));
    const auto jy = back((f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8]));
    const auto inv_rho = recip(rho);
    const auto ux = fmul(FORCE ? ffma(half, p.Fx, jx) : jx, inv_rho);
    const auto uy = fmul(jy, inv_rho);
    const auto bx = back(((gx[0] + gx[1]) + (gx[2] + gx[3])) + gx[4]);
    const auto dby = back(((gy[0] + gy[1]) + (gy[2] + gy[3])) + gy[4]);
    const auto by = p.B0 + dby;
    const auto q = fmul(dby, p.B0 + by);
    const auto om13 = fmul(p.owf1, fmul(2.25f, ffma(-bx, bx, q)));
    const auto omxy = fmul(p.owf5, fmul(fmul(9.0f, bx), by));
    const auto usq = fmul(one5, ffma(ux, ux, fmul(uy, uy)));
    V s0 = zero_of<V>(), s1p = s0, s1z = s0, s1m = s0, s5p = s0, s5m = s0;  // source prefactors
    if constexpr (FORCE) {
        s0 = fmul(p.sw0, -ux);
        s1p = fmul(p.sw1, 1.0f - ux), s1z = fmul(p.sw1, -ux), s1m = fmul(p.sw1, -1.0f - ux);
        s5p = fmul(p.sw5, 1.0f - ux), s5m = fmul(p.sw5, -1.0f - ux);
    }
    auto dir = [&](int a, V eu, float ow, V omag, V sa) {
        const auto bm1 = ffma(ffma(four5, eu, three), eu, -usq);
        const auto ofeq = ffma(ow, ffma(rho, bm1, drho), omag);
        if constexpr (FORCE)
            f[a] = ffma(p.om1f, f[a], ofeq + ffma(sa, bm1, sa));
        else
            f[a] = ffma(p.om1f, f[a], ofeq);
    };
    const V zero = zero_of<V>();
    dir(0, zero, p.owf0, zero, s0);
    dir(1, ux, p.owf1, om13, s1p);
    dir(2, uy, p.owf1, -om13, s1z);
    dir(3, -ux, p.owf1, om13, s1m);
    dir(4, -uy, p.owf1, -om13, s1z);
    dir(5, ux + uy, p.owf5, -omxy, s5p);
    dir(6, uy - ux, p.owf5, omxy, s5m);
    dir(7, -ux - uy, p.owf5, -omxy, s5m);
    dir(8, ux - uy, p.owf5, omxy, s5p);
    collide_g<float>(gx, gy, ux, uy, bx, by, dby, p);
}

// Moment closure and collision of a thread's node or nodes.  A scaled row is closed unscaled.
template <int CLOSURE, int COUPLING, bool FORCE, bool SCALED, typename V>
__device__ __forceinline__ void close_collide(V f[9], V gx[5], V gy[5], const StepParams<float>& p, bool bottom,
                                              bool top) {
    if constexpr (COUPLING == 1) {
        if constexpr (std::is_same<V, float>::value) {
            if (CLOSURE == 1 && bottom) moment_closure_bottom<float, 1>(f, gx, gy, p.bot, p);
            if (CLOSURE == 1 && top) moment_closure_top<float, 1>(f, gx, gy, p.top, p);
            collide<float, 1>(f, gx, gy, p);
        } else {
            close_collide_pair<CLOSURE, 1, true>(f, gx, gy, p, bottom, top);
        }
    } else {
        if (CLOSURE == 1 && (bottom || top)) {
            auto all = [&](float c) {
#pragma unroll
                for (int a = 0; a < 9; ++a) f[a] = fmul(c, f[a]);
#pragma unroll
                for (int a = 0; a < 5; ++a) gx[a] = fmul(c, gx[a]), gy[a] = fmul(c, gy[a]);
            };
            if (SCALED) all(kHalfUnscale);
            if (bottom) moment_closure_bottom<float, 0>(f, gx, gy, p.bot, p);
            if (top) moment_closure_top<float, 0>(f, gx, gy, p.top, p);
            if (SCALED) all(kHalfScale);
        }
        collide_rows<FORCE, SCALED>(f, gx, gy, p);
    }
}

// What a thread keeps of a level for the next one, as storage words: of the row before, the e_x = 0
// populations (f0, gx0, gy0; f2, gx2, gy2; and, for a bottom link wall, f4, gx4, gy4), and of the
// row before that the upward ones (f2, gx2, gy2; f5, f6 as the node pulls them).
template <typename W>
struct Kept {
    W a0[3], a2[3], a4[3], b2[3], b5, b6;
};

__device__ __forceinline__ int ey9(int a) {
    return a == 2 || a == 5 || a == 6 ? 1 : (a == 4 || a == 7 || a == 8 ? -1 : 0);
}
__device__ __forceinline__ int ey5(int a) { return a == 2 ? 1 : (a == 4 ? -1 : 0); }

// The planes of both buffers (f0..8, gx0..4, gy0..4).  As kernel parameters their addresses are uniform
// operands of the loads and stores, to which a thread adds 32-bit offsets: computing 64-bit addresses
// took 40 of 296 instructions per node and step.
struct RowPlanes {
    const char* in[19];
    char* out[19];
    // in place: what a block pulls from rows and columns of other blocks, saved before the pass
    const void *rows, *cols;
};

// Words of the in-place workspace: for each chunk boundary 2 T rows around it, [boundary][plane][2 T][ncol], then for
// each strip boundary 2 T columns, [strip][plane][ny][2 T].
struct RowHalos {
    int chunks, strips;
    int64_t rows, cols;
    __host__ __device__ RowHalos(int ncol, int ny, const RowsPlan& rp) {
        strips = (ncol + rp.strip - 1) / rp.strip;
        chunks = rp.edge >= ny ? 1 : 1 + (ny - rp.edge + rp.chunk - 1) / rp.chunk;
        rows = (int64_t)(chunks - 1) * 19 * (2 * kRowSteps) * ncol;
        cols = (int64_t)strips * 19 * (2 * kRowSteps) * ny;
    }
};

// Ring entries of a level: f1 f3 gx1 gx3 gy1 gy3 f5 f6 f7 f8 (the populations with e_x != 0).
constexpr int kRing = 10;

template <typename S, typename N, int CLOSURE, int COUPLING, bool FORCE, bool INPLACE, int T, int TB, int MINB>
__global__ void __launch_bounds__(TB, MINB) rows_kernel(const __grid_constant__ RowPlanes io,
                                                        const __grid_constant__ StepParams<float> p, int strip,
                                                        int chunk, int edge) {
    typedef typename N::W W;
    typedef typename N::V V;
    extern __shared__ __align__(16) unsigned char rows_sm[];
    const int t = threadIdx.x;
    const int ncol = p.nx / N::kNodes, ny = p.ny;   // columns of words
    const unsigned pitch = (unsigned)ncol * (unsigned)sizeof(W);  // bytes of a row
    const int x0 = blockIdx.x * strip, w = min(strip, ncol - x0);
    const bool wrap = !INPLACE && strip >= ncol;    // the whole row in one block
    const int halo = wrap ? 0 : T - 1;
    // The thread's slot among the block's columns.  In place the columns that pull from other blocks, three at each
    // end, go to the first warp, so that one warp takes the longer way to its words.
    const int slots = w + 2 * halo;
    const int sl = !INPLACE || slots <= 32 ? t : (t < 29 || t >= slots ? t : (t < 32 ? slots - 32 + t : t - 3));
    const bool lane = t < slots;
    const int u = lane ? x0 - halo + sl : x0;  // the thread's column, beyond the periodic edge in a halo
    int c = u;
    if (c < 0) c += ncol;
    if (c >= ncol) c -= ncol;
    const unsigned cl = (c == 0 ? ncol - 1 : c - 1) * sizeof(W), cc = c * sizeof(W),
                   cr = (c == ncol - 1 ? 0 : c + 1) * sizeof(W);
    // the neighbouring columns' slots in shared memory, relative to the own one
    const int dl = wrap && t == 0 ? w - 1 : (sl == 0 ? 0 : -1);
    const int dr = wrap && t == w - 1 ? 1 - w : (sl == TB - 1 ? 0 : 1);
    const bool mine = lane && sl >= halo && sl < halo + w;
    // chunk 0 and the last one, which take the slower path with the walls, are shorter: edge rows
    const int y0 = blockIdx.y == 0 ? 0 : edge + (blockIdx.y - 1) * chunk;
    const int y1 = blockIdx.y == 0 ? min(edge, ny) : min(ny, y0 + chunk);

    // ring slots of this row, the row before and the one before that: slot s of level k, entry v is
    // base + ((k - 1) * 3 + s) * kRing * TB + v * TB
    constexpr int kLevel = 3 * kRing * TB;
    W* q0 = reinterpret_cast<W*>(rows_sm) + sl;
    W* q1 = q0 + kRing * TB;
    W* q2 = q1 + kRing * TB;
    Kept<W> kept[T - 1] = {};

    // In place, near a block's edge: where the planes' words of column v (beyond the periodic edge or not) of row y
    // are, in the saved copy if the row or the column is another block's: plane a < 9 at f + a ps, 9 + a at g + a ps.
    // Selects rather than a branch per load, which would wait for each load.
    struct Planes {
        const char *f, *g;
        unsigned ps;
    };
    auto planes_at = [&](int y, int v) -> Planes {
        Planes q;
        if (y < y0 || y >= y1) {  // the same for the whole block
            const int vm = v < 0 ? v + ncol : (v >= ncol ? v - ncol : v);
            const int b = (int)blockIdx.y - (y < y0 ? 1 : 0), k = y - (y < y0 ? y0 : y1) + T;
            q.ps = 2 * T * pitch;
            q.f = (const char*)io.rows +
                  ((uint64_t)(unsigned)(b * 19) * q.ps + (unsigned)k * pitch + vm * (unsigned)sizeof(W));
            q.g = q.f + 9 * (uint64_t)q.ps;
            return q;
        }
        const bool left = v < x0, out = left || v >= x0 + w;
        const int b = left ? blockIdx.x : (blockIdx.x + 1 == gridDim.x ? 0 : blockIdx.x + 1);
        const unsigned saved = 2 * T * sizeof(W) * ny, plane = pitch * ny;
        const unsigned at_out = (unsigned)y * (2 * T * sizeof(W)) +
                                (v - (left ? x0 : x0 + w) + T) * (unsigned)sizeof(W);
        const unsigned at_own = (unsigned)y * pitch + v * (unsigned)sizeof(W);
        const char* base = (const char*)io.cols + (uint64_t)(unsigned)(b * 19) * saved;
        const unsigned at = out ? at_out : at_own;
        q.ps = out ? saved : plane;
        q.f = (out ? base : io.in[0]) + at;
        q.g = (out ? base + 9 * (uint64_t)saved : io.in[9]) + at;
        return q;
    };
    // Row r: level 1 of row r, ..., level T of row r - (T - 1).  now / before: ring slots.
    auto row = [&](auto walls, int r, W* now, W* before) {
        // Without WALLS no level's row is beyond or at a wall; a level that is not on yet then computes
        // something nobody uses.
        constexpr bool WALLS = decltype(walls)::value;
        V f[9], gx[5], gy[5];
        W cur[9];  // words of the level just computed: f0 gx0 gy0, f2 gx2 gy2, f4 gx4 gy4
#pragma unroll
        for (int k = 1; k <= T; ++k) {
            const int j = r - (k - 1);  // this level's row
            const bool on = !WALLS || (j >= max(0, y0 - (T - k)) && j < min(ny, y1 + (T - k)));
            const bool bottom = WALLS && j == 0, top = WALLS && j == ny - 1;
            if (k == 1) {
                if (on) {
                    // get(plane, dy, dx): the word of the own column + dx in row j + dy
                    auto load = [&](auto get) {
                        auto same = [&](int a, int dy) -> V { return N::unpack(get(a, dy, 0)); };
                        auto left = [&](int a, int dy) -> V {
                            return N::unpack(N::from_left(get(a, dy, -1), N::kOwn ? get(a, dy, 0) : W()));
                        };
                        auto right = [&](int a, int dy) -> V {
                            return N::unpack(N::from_right(N::kOwn ? get(a, dy, 0) : W(), get(a, dy, 1)));
                        };
                        f[0] = same(0, 0);
                        f[1] = left(1, 0);
                        f[3] = right(3, 0);
                        gx[0] = same(9, 0);
                        gx[1] = left(10, 0);
                        gx[3] = right(12, 0);
                        gy[0] = same(14, 0);
                        gy[1] = left(15, 0);
                        gy[3] = right(17, 0);
                        if (!bottom) {
                            f[2] = same(2, -1);
                            f[5] = left(5, -1);
                            f[6] = right(6, -1);
                            gx[2] = same(11, -1);
                            gy[2] = same(16, -1);
                        } else if (CLOSURE == 0) {  // the node's own outgoing populations
                            f[2] = same(4, 0);
                            f[5] = same(7, 0);
                            f[6] = same(8, 0);
                            gx[2] = same(13, 0);
                            gy[2] = same(18, 0);
                        }
                        if (!top) {
                            f[4] = same(4, 1);
                            f[7] = right(7, 1);
                            f[8] = left(8, 1);
                            gx[4] = same(13, 1);
                            gy[4] = same(18, 1);
                        } else if (CLOSURE == 0) {
                            f[4] = same(2, 0);
                            f[7] = same(5, 0);
                            f[8] = same(6, 0);
                            gx[4] = same(11, 0);
                            gy[4] = same(16, 0);
                        }
                    };
                    const unsigned rc = (unsigned)j * pitch, rs = rc - pitch, rn = rc + pitch;  // bytes
                    auto near = [&](int a, int dy, int dx) -> W {
                        const W* q = reinterpret_cast<const W*>(io.in[a] + ((dy == 0 ? rc : (dy < 0 ? rs : rn)) +
                                                                             (dx == 0 ? cc : (dx < 0 ? cl : cr))));
                        return INPLACE ? *q : __ldg(q);
                    };
                    if constexpr (INPLACE) {
                        if (__all_sync(0xffffffffu, u > x0 && u + 1 < x0 + w && j > y0 && j + 1 < y1))
                            load(near);
                        else
                            load([&](int a, int dy, int dx) -> W {
                                const Planes q = planes_at(j + dy, u + dx);
                                return *reinterpret_cast<const W*>((a < 9 ? q.f : q.g) +
                                                                   (uint64_t)q.ps * (a < 9 ? a : a - 9));
                            });
                    } else {
                        load(near);
                    }
                }
            } else {
                // the level before: row j + 1 in `cur` and slot `now`, row j in `kept` and slot `before`
                W *rn = now + (k - 2) * kLevel, *rb = before + (k - 2) * kLevel;
                const W *rnl = rn + dl, *rnr = rn + dr, *rbl = rb + dl, *rbr = rb + dr;
                auto left = [&](const W* q, const W* ql, int v) -> W {
                    return N::from_left(ql[v * TB], N::kOwn ? q[v * TB] : W());
                };
                auto right = [&](const W* q, const W* qr, int v) -> W {
                    return N::from_right(N::kOwn ? q[v * TB] : W(), qr[v * TB]);
                };
                Kept<W>& K = kept[k - 2];
                if (on) {
                    f[0] = N::unpack(K.a0[0]);
                    gx[0] = N::unpack(K.a0[1]);
                    gy[0] = N::unpack(K.a0[2]);
                    f[1] = N::unpack(left(rb, rbl, 0));
                    f[3] = N::unpack(right(rb, rbr, 1));
                    gx[1] = N::unpack(left(rb, rbl, 2));
                    gx[3] = N::unpack(right(rb, rbr, 3));
                    gy[1] = N::unpack(left(rb, rbl, 4));
                    gy[3] = N::unpack(right(rb, rbr, 5));
                    if (!bottom) {
                        f[2] = N::unpack(K.b2[0]);
                        gx[2] = N::unpack(K.b2[1]);
                        gy[2] = N::unpack(K.b2[2]);
                        f[5] = N::unpack(K.b5);
                        f[6] = N::unpack(K.b6);
                    } else if (CLOSURE == 0) {
                        f[2] = N::unpack(K.a4[0]);
                        gx[2] = N::unpack(K.a4[1]);
                        gy[2] = N::unpack(K.a4[2]);
                        f[5] = N::unpack(rb[8 * TB]);
                        f[6] = N::unpack(rb[9 * TB]);
                    }
                    if (!top) {
                        f[4] = N::unpack(cur[6]);
                        gx[4] = N::unpack(cur[7]);
                        gy[4] = N::unpack(cur[8]);
                        f[7] = N::unpack(right(rn, rnr, 8));
                        f[8] = N::unpack(left(rn, rnl, 9));
                    } else if (CLOSURE == 0) {
                        f[4] = N::unpack(K.a2[0]);
                        gx[4] = N::unpack(K.a2[1]);
                        gy[4] = N::unpack(K.a2[2]);
                        f[7] = N::unpack(rb[6 * TB]);
                        f[8] = N::unpack(rb[7 * TB]);
                    }
                }
                // the level before moves up one row
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    K.b2[q] = K.a2[q];
                    K.a0[q] = cur[q];
                    K.a2[q] = cur[3 + q];
                    if (CLOSURE == 0) K.a4[q] = cur[6 + q];
                }
                K.b5 = left(rb, rbl, 6);
                K.b6 = right(rb, rbr, 7);
            }
            if (on) {
                if (CLOSURE == 0) {
                    if (bottom) {
                        f[5] = f[5] + p.bot.du;
                        f[6] = f[6] - p.bot.du;
                        gx[2] = ffma(p.bot.r, gx[2], p.bot.kx);
                        gy[2] = -gy[2];
                    }
                    if (top) {
                        f[7] = f[7] - p.top.du;
                        f[8] = f[8] + p.top.du;
                        gx[4] = ffma(p.top.r, gx[4], p.top.kx);
                        gy[4] = -gy[4];
                    }
                }
                close_collide<CLOSURE, COUPLING, FORCE, IsScaled<N>::value>(f, gx, gy, p, bottom, top);
                if (k < T) {
                    W* ring = now + (k - 1) * kLevel;
                    const V x[kRing] = {f[1], f[3], gx[1], gx[3], gy[1], gy[3], f[5], f[6], f[7], f[8]};
#pragma unroll
                    for (int v = 0; v < kRing; ++v) ring[v * TB] = N::pack(x[v]);
                    const V own[9] = {f[0], gx[0], gy[0], f[2], gx[2], gy[2], f[4], gx[4], gy[4]};
#pragma unroll
                    for (int q = 0; q < 9; ++q) cur[q] = N::pack(own[q]);
                } else if (mine && (WALLS || j >= y0)) {
                    const unsigned n = (unsigned)j * pitch + cc;
                    auto put = [&](int a, V v) {
                        *reinterpret_cast<W*>(io.out[a] + n) = N::pack(v);
                    };
#pragma unroll
                    for (int a = 0; a < 9; ++a) put(a, f[a]);
#pragma unroll
                    for (int a = 0; a < 5; ++a) put(9 + a, gx[a]);
#pragma unroll
                    for (int a = 0; a < 5; ++a) put(14 + a, gy[a]);
                }
            }
            if (k < T) __syncthreads();
        }
    };

    // The row that iteration r + kAhead will be the first to pull, brought into L2 (one line of one plane
    // per thread).
    const int lines = (w + 2 * halo) * (int)sizeof(W) / 128 + 1, pa = t / lines;
    const int pey = pa < 9 ? ey9(pa) : ey5(pa < 14 ? pa - 9 : pa - 14);
    const int px = x0 - halo < 0 ? 0 : x0 - halo;
    const char* pf = io.in[min(pa, 18)] +
                     min((px + (t % lines) * (128 / (int)sizeof(W))), ncol - 1) * (int)sizeof(W);
    auto prefetch = [&](int r) {
        const int y = r + kAhead - pey;
        if (pa < 19 && y >= 0 && y < ny)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(pf + (uint64_t)((unsigned)y * pitch)));
    };
    auto up = [&]() {  // the slots move up one row
        W* q = q0;
        q0 = q1;
        q1 = q2;
        q2 = q;
    };
    const int last = y1 - 1 + (T - 1);
    if (y0 >= T && y1 <= ny - T) {
#pragma unroll 1
        for (int r = y0 - (T - 1); r <= last; ++r) {
            prefetch(r);
            row(std::false_type{}, r, q0, q2);
            up();
        }
    } else {
#pragma unroll 1
        for (int r = max(0, y0 - (T - 1)); r <= last; ++r) {
            row(std::true_type{}, r, q0, q2);
            up();
        }
    }
}

// Copies the rows and columns around the blocks' boundaries (RowHalos) before an in-place pass overwrites them.
// blockIdx.x: boundary and plane; blockIdx.y: a part of it.
template <typename W>
__global__ void __launch_bounds__(256) rows_save_kernel(const __grid_constant__ RowPlanes io, int ncol, int ny,
                                                        const __grid_constant__ RowsPlan rp, W* rows, W* cols) {
    constexpr int D = 2 * kRowSteps;
    const RowHalos h(ncol, ny, rp);
    const int a = blockIdx.x % 19, b = blockIdx.x / 19;
    const int first = blockIdx.y * blockDim.x + threadIdx.x, stride = gridDim.y * blockDim.x;
    const W* in = reinterpret_cast<const W*>(io.in[a]);
    if (b < h.chunks - 1) {
        const int y = rp.edge + b * rp.chunk - kRowSteps, n = min(D, ny - y);  // a last chunk may be shorter
        const W* src = in + (int64_t)y * ncol;
        W* dst = rows + (int64_t)(b * 19 + a) * D * ncol;
        for (int k = first; k < n * ncol; k += stride) dst[k] = src[k];
    } else {
        const int s = b - (h.chunks - 1);
        W* dst = cols + (int64_t)(s * 19 + a) * ny * D;
        for (int k = first; k < D * ny; k += stride) {
            const int y = k / D, v = s * rp.strip - kRowSteps + (k - y * D);
            dst[k] = in[(int64_t)y * ncol + (v < 0 ? v + ncol : (v >= ncol ? v - ncol : v))];
        }
    }
}

template <typename S, typename N, bool INPLACE, int TB, int MINB>
struct Rows {
    static constexpr int kThreads = TB, kNodes = N::kNodes;
    // the Maxwell coupling's form of the node type
    static constexpr bool kScaled = std::is_same<N, TwoNodes<__half>>::value;
    typedef typename std::conditional<kScaled, TwoNodesScaled<S>, N>::type M;
    static constexpr bool kInplace = INPLACE;
    typedef void (*Fn)(const RowPlanes, const StepParams<float>, int, int, int);
    template <int CLOSURE, int COUPLING>
    static Fn typed(bool force) {
        typedef typename std::conditional<COUPLING == 0, M, N>::type K;
        if constexpr (COUPLING == 0)
            if (!force) return rows_kernel<S, K, CLOSURE, 0, false, INPLACE, kRowSteps, TB, MINB>;
        return rows_kernel<S, K, CLOSURE, COUPLING, true, INPLACE, kRowSteps, TB, MINB>;
    }
    static Fn kernel(int closure, int coupling, bool force) {
        if (coupling == 0) return closure == 0 ? typed<0, 0>(force) : typed<1, 0>(force);
        return closure == 0 ? typed<0, 1>(force) : typed<1, 1>(force);
    }
    static constexpr size_t smem() { return (size_t)(kRowSteps - 1) * 3 * kRing * TB * sizeof(typename N::W); }
    static cudaError_t prepare(int closure, int coupling, bool force, int* blocks) {
        Fn k = kernel(closure, coupling, force);
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem());
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, k, TB, smem());
        return e;
    }
    static void launch(const void* fin, const void* gin, void* fout, void* gout, const StepParams<float>& p,
                       int closure, const RowsPlan& rp, void* work, cudaStream_t st) {
        const int ncol = p.nx / N::kNodes;
        const RowHalos halos(ncol, p.ny, rp);
        const dim3 grid(halos.strips, halos.chunks);
        RowPlanes io;
        for (int a = 0; a < 19; ++a) {
            io.in[a] = (const char*)(a < 9 ? (const S*)fin + a * p.N : (const S*)gin + (a - 9) * p.N);
            io.out[a] = (char*)(a < 9 ? (S*)fout + a * p.N : (S*)gout + (a - 9) * p.N);
        }
        io.rows = io.cols = nullptr;
        if (INPLACE) {
            typedef typename N::W W;
            W *rows = (W*)work, *cols = rows + halos.rows;
            rows_save_kernel<W><<<dim3(19 * (halos.chunks - 1 + halos.strips), 8), 256, 0, st>>>(io, ncol, p.ny, rp,
                                                                                                rows, cols);
            io.rows = rows;
            io.cols = cols;
        }
        kernel(closure, p.coupling, p.Fx != 0.0f)<<<grid, TB, smem(), st>>>(
            io, kScaled && p.coupling == 0 ? scaled_params(p, closure) : p, rp.strip, rp.chunk, rp.edge);
    }
};
// Threads per block and blocks per SM, timed at 4096^2 (GLUPS, moment closure): FP32 128 x 5 98, 128 x 6 93,
// 192 x 4 98, 256 x 3 91, 320 x 2 92; BF16 128 x 4 126, 96 x 5 118, 256 x 2 113, 128 x 5 98 (spills).  Small
// blocks wait less at their barriers; the extra columns of narrow strips cost more below 128.
#define F32S 128, 5
#define H16S 128, 4
typedef Rows<float, OneNode<float>, false, F32S> RowsF32;
typedef Rows<__nv_bfloat16, TwoNodes<__nv_bfloat16>, false, H16S> RowsBf16;
typedef Rows<__half, TwoNodes<__half>, false, H16S> RowsF16;
typedef Rows<float, OneNode<float>, true, F32S> InplaceF32;

}  // namespace

// Strips and chunks of the kernel R: as many blocks as are resident at once.
template <typename R>
static cudaError_t plan_typed(int closure, int coupling, bool force, int nx, int ny, double least, RowsPlan* rp) {
    int dev = 0, sms = 0, blocks = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = R::prepare(closure, coupling, force, &blocks);
    if (e != cudaSuccess) return e;
    const int ncol = nx / R::kNodes;
    const int most = R::kThreads - 2 * (kRowSteps - 1);
    int strips = 1, strip = ncol;
    if (ncol > (R::kInplace ? most : R::kThreads)) {
        strips = (ncol + most - 1) / most;
        strip = std::min(most, ((ncol + strips - 1) / strips + 7) / 8 * 8);
        strips = (ncol + strip - 1) / strip;
    }
    const int slots = std::max(1, sms * blocks / strips);
    // chunks of `chunk` rows and one of `edge` rows at each wall: 2 edge + (slots - 2) chunk >= ny
    int chunk = (ny + slots - 1) / slots, edge = chunk;
    if (slots >= 3) {
        chunk = (int)((ny + slots - 2 * kEdgeShare) / (slots - 2 + 2 * kEdgeShare));
        for (;; ++chunk) {
            edge = std::max(kRowSteps, (int)(kEdgeShare * chunk));
            if (2 * (int64_t)edge + (int64_t)(slots - 2) * chunk >= ny) break;
        }
    }
    const double use = (double)nx * ny / ((double)slots * strips * R::kThreads * R::kNodes * (chunk + kRowSteps - 1));
    if (chunk < kRowMinChunk || use < least) return cudaSuccess;
    rp->strip = strip;
    rp->chunk = chunk;
    rp->edge = edge;
    return cudaSuccess;
}

cudaError_t plan_rows(int storage, int closure, const StepParams<double>& p, int inplace, RowsPlan* rp) {
    const int nx = p.nx, ny = p.ny, coupling = p.coupling;
    const bool force = (float)p.Fx != 0.0f;
    rp->strip = rp->chunk = rp->edge = 0;
    if (storage == 0 || (storage >= 2 && nx % 2 != 0) || nx < 64) return cudaSuccess;
    int dev = 0, l2 = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
    if (e != cudaSuccess) return e;
    const bool memory = (int64_t)(inplace ? 19 : 38) * storage_bytes(storage) * nx * ny > l2;
    if (inplace) {
        // FP32 only: the interleaved rows of 16-bit storage ran at 64 (BF16) and 58 (FP16) GLUPS at 2056 x 1500
        // against 72 and 71 in AA pairs.  Plane strides are 32-bit.
        if (storage != 1 || !memory || (int64_t)nx * ny * 4 >= (int64_t)1 << 32) return cudaSuccess;
        return plan_typed<InplaceF32>(closure, coupling, force, nx, ny, kUseInPlace, rp);
    }
    const double least = memory ? kUseMemory : kUseL2;
    if (storage == 1) return plan_typed<RowsF32>(closure, coupling, force, nx, ny, least, rp);
    if (storage == 2) return plan_typed<RowsBf16>(closure, coupling, force, nx, ny, least, rp);
    return plan_typed<RowsF16>(closure, coupling, force, nx, ny, least, rp);
}

size_t rows_workspace(int nx, int ny, const RowsPlan& rp) {
    const RowHalos h(nx, ny, rp);
    return (size_t)(h.rows + h.cols) * sizeof(float);
}

cudaError_t launch_rows(int storage, int closure, const void* fin, const void* gin, void* fout, void* gout,
                        const StepParams<double>& pd, const RowsPlan& rp, void* work, cudaStream_t st) {
    const StepParams<float> p = convert_params<float>(pd);
    if (work) InplaceF32::launch(fin, gin, fout, gout, p, closure, rp, work, st);
    else if (storage == 1) RowsF32::launch(fin, gin, fout, gout, p, closure, rp, nullptr, st);
    else if (storage == 2) RowsBf16::launch(fin, gin, fout, gout, p, closure, rp, nullptr, st);
    else RowsF16::launch(fin, gin, fout, gout, p, closure, rp, nullptr, st);
    return cudaGetLastError();
}

}  // namespace lks
