// lks_step_staged.cu -- the fused step of one lattice with 16-bit deviation storage, rows staged
// through shared memory by the bulk-copy engine (two-buffer handles; nx a multiple of 8 and at least
// kSegX).  The pull, wall closures, collision and store as in step_node_with (lks_device.cuh), with the same per-node
// arithmetic: the results agree bit for bit with the one- and two-node kernels.
//
// A task is a row segment of up to kSegX nodes (x0 .. x0 + T - 1 of row y), the segments of a row of equal
// length.  For each of the 19 population slots (f_0..8, g_x0..4, g_y0..4) a producer warp copies, one slot
// per lane, the segment of the row the slot pulls from (y - e_y; a link-closure wall row takes its own row
// of the opposite plane; a moment-closure wall row fetches nothing for the slots it reconstructs) into one
// of the shared-memory stages, with a 16-byte halo on each side for the x-shifted slots (periodic in x:
// wrapped copies at the row ends), completing on the stage's `full` mbarrier.  The consumer warps take
// the tasks' nodes 64 at a time (lks_ring.cuh): a lane reads 19 words (two x-adjacent nodes; byte_perm for the x
// shift) into registers, the warp arrives on the stage's `empty` mbarrier, so that the producer refills it
// while the warp computes, and then come the wall closure, the collision as one float2 (packed FP32x2
// arithmetic) and 19 packed words stored.  Rows without a wall run a path with no closure code.  Every
// wait is bounded (kWaitNs); one that runs out sets *err and ends that warp's loop, and the producer
// waits, within the same limit, for its last copies to each stage before it returns.
//
// Bound by memory (76 bytes a node and step) and by how evenly the block's warps are kept at it.  With
// sixteen warps tied to the sixteen 64-node shares of a task, a row of 2056 nodes left a third of the
// tasks four words long; and 17 warps have 96 registers, too few to hold the words, so they went through
// a scratch area.  Fifteen warps and the producer have 128.  Three stages: two starve the warps, four and
// five put more reads among the writes than DRAM likes.  us a step, before -> after: BF16 in place
// 2056 x 1500 47.8 -> 43.1, 4096^2 206 -> 203 (two stages 223, five 214.5), 3000^2 113.9 -> 112.9 (126, 118); two
// buffers BF16 1024 x 1000 16.1 -> 15.3, 4096 x 150 10.7 -> 10.2, 2056 x 400 FP16 16.8 -> 14.6.  A warp's wait for the
// tasks it has no item in is among these times (1 % of them at 11 items a task).
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "lks_bulk.cuh"
#include "lks_device.cuh"
#include "lks_internal.h"
#include "lks_packed.cuh"
#include "lks_pair.cuh"
#include "lks_pdl.cuh"
#include "lks_ring.cuh"

namespace lks {
namespace {

constexpr int kSegX = 1024;                      // nodes of a task, at most
constexpr int kHaloW = 4;                        // halo words (8 elements = 16 bytes) per side
constexpr int kSlotW = kSegX / 2 + 2 * kHaloW;   // words of a staged slot row
constexpr int kSlots = 19;
constexpr int kStages = 3;
constexpr int kStageW = kSlots * kSlotW;
constexpr int kConsumerWarps = 15;
constexpr int kThreads = (kConsumerWarps + 1) * 32;  // consumers + the producer warp
constexpr uint64_t kWaitNs = 1000000000ull;      // 1 s
constexpr size_t kSmem = 128 + (size_t)kStages * kStageW * 4;
static_assert(kSmem <= 227 * 1024, "shared memory per block");

// The destination planes: a store adds one 32-bit offset to a uniform base.
struct SlotPlanes {
    void* slot[kSlots];
};
__device__ __forceinline__ void put_word(const SlotPlanes& d, int k, uint32_t byte, uint32_t v) {
    *reinterpret_cast<uint32_t*>(static_cast<char*>(d.slot[k]) + byte) = v;
}

// Segments of a row: as few as kSegX allows, of equal length in items (64 nodes, or 32 words).
struct Segments {
    int n, items;  // segments per row, items per segment
};
inline Segments segments_of(int nx) {
    const int n = (nx + kSegX - 1) / kSegX;
    return {n, ((nx + n - 1) / n + 63) / 64};
}

// The row and segment of task t0 + k G, for k = 0, 1, ... in order.
struct TaskAt {
    uint32_t k;
    int y, g;  // row, segment
    __device__ __forceinline__ explicit TaskAt(int nseg) : k(0), y(blockIdx.x / nseg), g(blockIdx.x % nseg) {}
    __device__ __forceinline__ void to(uint32_t it, int nseg, int dy, int dg) {
        for (; k < it; ++k) {
            y += dy;
            g += dg;
            if (g >= nseg) g -= nseg, ++y;
        }
    }
};

// A consumer warp's part in a task in which it has no item (lks_ring.cuh).
__device__ __forceinline__ bool pass_task(uint64_t* full, uint64_t* empty, uint32_t it, int lane, int* err) {
    const uint32_t s = it % kStages;
    if (!mbar_wait_bounded(&full[s], (it / kStages) & 1u, kWaitNs)) {
        atomicExch(err, 1);
        return false;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    return true;
}

// D2Q9 (f) and D2Q5 (g) directions of slot k: k < 9 is f_k, 9..13 is g_x,k-9, 14..18 is g_y,k-14.
__host__ __device__ constexpr int dir_of(int k) { return k < 9 ? k : (k < 14 ? k - 9 : k - 14); }
__host__ __device__ constexpr int ex9(int a) {
    return (a == 1 || a == 5 || a == 8) ? 1 : (a == 3 || a == 6 || a == 7) ? -1 : 0;
}
__host__ __device__ constexpr int ey9(int a) {
    return (a == 2 || a == 5 || a == 6) ? 1 : (a == 4 || a == 7 || a == 8) ? -1 : 0;
}
__host__ __device__ constexpr int opp9(int a) { return a == 0 ? 0 : (a <= 4 ? (a + 1) % 4 + 1 : (a + 1) % 4 + 5); }
// plane of slot k's population table for direction a (f: a; g_x: a; g_y: 5 + a)
__host__ __device__ constexpr int plane_of(int k, int a) { return k < 9 ? a : (k < 14 ? a : 5 + a); }

template <typename S, int CLOSURE, int COUPLING>
__global__ void __launch_bounds__(kThreads, 1) step_kernel_staged(const S* __restrict__ fin, const S* __restrict__ gin,
                                                                   const SlotPlanes out, const StepParams<float> p,
                                                                   const Segments sg, int* err) {
    extern __shared__ __align__(128) unsigned char sm[];
    uint64_t* full = reinterpret_cast<uint64_t*>(sm);
    uint64_t* empty = full + kStages;
    uint32_t* stage0 = reinterpret_cast<uint32_t*>(sm + 128);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nx = p.nx, ny = p.ny;
    const int64_t N = p.N;
    const int nseg = sg.n, seg = 64 * sg.items;
    const int64_t ntask = (int64_t)ny * nseg;
    const int64_t G = gridDim.x, t0 = blockIdx.x;
    const int64_t nmine = t0 < ntask ? (ntask - 1 - t0) / G + 1 : 0;  // tasks t0, t0 + G, ...
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], ring_arrivals(sg.items, kConsumerWarps));
        }
        mbar_init_fence();
    }
    pdl_wait();
    __syncthreads();

    if (warp == kConsumerWarps) {  // producer: lane k < 19 fetches slot k
        const int k = lane < kSlots ? lane : 0;
        const int a = dir_of(k), ex = ex9(a), ey = ey9(a);
        const S* base = k < 9 ? fin : gin;
        const S* bn = base + (int64_t)plane_of(k, a) * N;        // the slot's own direction
        const S* bw = base + (int64_t)plane_of(k, opp9(a)) * N;  // the opposite one (link walls)
        int64_t it = 0;
        for (; it < nmine; ++it) {
            const int s = (int)(it % kStages);
            const int64_t u = it / kStages;
            if (u > 0 && !mbar_wait_bounded(&empty[s], (uint32_t)(u - 1) & 1u, kWaitNs)) {
                if (lane == 0) atomicExch(err, 1);
                break;
            }
            const int64_t t = t0 + it * G;
            const int y = (int)(t / nseg), x0 = (int)(t % nseg) * seg;
            const int T = min(seg, nx - x0);
            const bool wall = (ey == 1 && y == 0) || (ey == -1 && y == ny - 1);
            uint32_t* dst = stage0 + s * kStageW + k * kSlotW;
            // this lane's copies: (global element offset, shared word offset, elements)
            int64_t g0 = 0, g1 = 0, g2 = 0;
            int w0 = 0, w1 = 0, w2 = 0, n0 = 0, n1 = 0, n2 = 0;
            if (lane < kSlots) {
                if (wall) {
                    if (CLOSURE == 0) {  // link: own row, opposite plane
                        g0 = (int64_t)y * nx + x0;
                        w0 = kHaloW;
                        n0 = T;
                    }
                } else {
                    const int64_t row = (int64_t)(y - ey) * nx;
                    if (ex == 0) {
                        g0 = row + x0, w0 = kHaloW, n0 = T;
                    } else if (x0 >= 8 && x0 + T + 8 <= nx) {  // both halos in one copy
                        g0 = row + x0 - 8, w0 = 0, n0 = T + 16;
                    } else {
                        g0 = row + x0, w0 = kHaloW, n0 = T;
                        if (ex == 1) g1 = row + (x0 == 0 ? nx - 8 : x0 - 8), w1 = 0, n1 = 8;
                        else g2 = row + (x0 + T == nx ? 0 : x0 + T), w2 = kHaloW + T / 2, n2 = 8;
                    }
                }
            }
            const uint32_t mine = 2u * (uint32_t)(n0 + n1 + n2);
            const uint32_t bytes = __reduce_add_sync(0xffffffffu, mine);
            if (lane == 0) mbar_arrive_expect_tx(&full[s], bytes);
            __syncwarp();
            const S* src = (wall && CLOSURE == 0) ? bw : bn;
            if (n0) bulk_g2s(dst + w0, src + g0, 2u * n0, &full[s]);
            if (n1) bulk_g2s(dst + w1, src + g1, 2u * n1, &full[s]);
            if (n2) bulk_g2s(dst + w2, src + g2, 2u * n2, &full[s]);
        }
        // no copy may be left in flight into this block's shared memory: wait for the last phase
        // issued to each stage (already complete unless a consumer gave up)
        for (int s = 0; s < kStages; ++s) {
            if (it <= s) continue;
            const int64_t u_last = (it - 1 - s) / kStages;
            if (!mbar_wait_bounded(&full[s], (uint32_t)u_last & 1u, kWaitNs) && lane == 0) atomicExch(err, 1);
        }
        return;
    }

    // consumers: of item c of a task, a lane holds nodes x0 + 64 c + 2 lane and the next
    typedef Packed<S> P;
    const int dy = (int)(G / nseg), dg = (int)(G % nseg);
    const auto skip = [&](uint32_t it) -> bool { return pass_task(full, empty, it, lane, err); };
    ItemWalk<kConsumerWarps> i(warp);
    TaskAt at(nseg);
    for (; i.next((uint32_t)nmine, sg.items, skip); i.c += kConsumerWarps) {
        at.to(i.it, nseg, dy, dg);
        const uint32_t s = i.it % kStages;
        if (!mbar_wait_bounded(&full[s], (i.it / kStages) & 1u, kWaitNs)) {
            atomicExch(err, 1);
            break;
        }
        const int y = at.y, x = at.g * seg + 64 * i.c + 2 * lane;
        const bool active = x < nx;
        {
            const bool bottom = (y == 0), top = (y == ny - 1);
            const uint32_t* st = stage0 + s * kStageW + kHaloW + 32 * i.c + lane;
            // rows without a wall (all but two) take a path with no closure code
            auto body = [&](auto walls) {
                constexpr bool W = decltype(walls)::value;
                uint32_t u[kSlots];
                if (active) {
#pragma unroll
                    for (int k = 0; k < kSlots; ++k) {
                        const int a = dir_of(k), ex = ex9(a), ey = ey9(a);
                        const bool wall = W && ((ey == 1 && bottom) || (ey == -1 && top));
                        const uint32_t* row = st + k * kSlotW;
                        if (wall || ex == 0)
                            u[k] = row[0];
                        else if (ex == 1)  // x <- x - 1 (high half of the word before), x + 1 <- x
                            u[k] = __byte_perm(row[-1], row[0], 0x5432);
                        else  // x <- x + 1, x + 1 <- x + 2 (low half of the word after)
                            u[k] = __byte_perm(row[0], row[1], 0x5432);
                    }
                }
                // the words are in registers: the stage goes back to the producer before the
                // collision and the stores
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[s]);
                if (!active) return;
                float2 v[kSlots];
#pragma unroll
                for (int k = 0; k < kSlots; ++k) v[k] = P::pair(u[k]);
                float2 f[9], gx[5], gy[5];
#pragma unroll
                for (int a = 0; a < 9; ++a) f[a] = v[a];
#pragma unroll
                for (int a = 0; a < 5; ++a) {
                    gx[a] = v[9 + a];
                    gy[a] = v[14 + a];
                }
                // wall closures (the link slots hold the node's own outgoing populations)
                if (W && CLOSURE == 0) {
                    if (bottom) {
                        const WallCoef<float>& w = p.bot;
                        f[5] = f[5] + w.du;
                        f[6] = f[6] - w.du;
                        gx[2] = ffma(w.r, gx[2], w.kx);
                        gy[2] = -gy[2];
                    }
                    if (top) {
                        const WallCoef<float>& w = p.top;
                        f[7] = f[7] - w.du;
                        f[8] = f[8] + w.du;
                        gx[4] = ffma(w.r, gx[4], w.kx);
                        gy[4] = -gy[4];
                    }
                }
                // moment closure, moments, equilibria and collision for both nodes
                close_collide_pair<CLOSURE, COUPLING, W>(f, gx, gy, p, bottom, top);
                const uint32_t q = 2u * ((uint32_t)y * nx + x);  // bytes: at most 2^30 nodes
#pragma unroll
                for (int a = 0; a < 9; ++a) put_word(out, a, q, P::pack(f[a].x, f[a].y));
#pragma unroll
                for (int a = 0; a < 5; ++a) put_word(out, 9 + a, q, P::pack(gx[a].x, gx[a].y));
#pragma unroll
                for (int a = 0; a < 5; ++a) put_word(out, 14 + a, q, P::pack(gy[a].x, gy[a].y));
            };
            if (bottom || top)
                body(std::true_type{});
            else
                body(std::false_type{});
        }
    }
}

// Phase 0 of the in-place pair of steps (lks_aa.cuh) for 16-bit storage, staged the same way.  The
// rows are interleaved (32-bit word w of a row holds nodes x = w and x = w + nx/2), so a shift by one
// node is a shift by one word, with the two halves swapped across the periodic row edge.  A task is
// up to kSegX/2 words of one row; the producer stages, for each slot, the words the task's nodes pull from
// (row y - e_y; link wall rows their own row of the opposite plane; moment wall rows nothing) with
// 16-byte halos as above.  Each consumer thread takes one word (two nodes), collides them as a
// float2 and pushes every direction b into plane bbar at x + e_b (a direction that would leave
// through a wall into its own plane b of its own word), as the pair kernel does.  Race freedom: the
// location a node pulls from in direction c, plane c at x - e_c, is written in this phase only by
// that node (its push of direction cbar), after its read; halo words a task stages but does not use
// belong to other nodes, and it never writes them.
template <typename S, int CLOSURE, int COUPLING>
__global__ void __launch_bounds__(kThreads, 1) step_kernel_aa_staged(const S* fb, const S* gb,
                                                                      const SlotPlanes out, const StepParams<float> p,
                                                                      const Segments sg, int* err) {
    extern __shared__ __align__(128) unsigned char sm[];
    uint64_t* full = reinterpret_cast<uint64_t*>(sm);
    uint64_t* empty = full + kStages;
    uint32_t* stage0 = reinterpret_cast<uint32_t*>(sm + 128);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ny = p.ny, H = p.nx / 2;              // words per row
    const int64_t NP = p.N / 2;                     // words per plane
    const int nseg = sg.n, segw = 32 * sg.items;
    const int64_t ntask = (int64_t)ny * nseg;
    const int64_t G = gridDim.x, t0 = blockIdx.x;
    const int64_t nmine = t0 < ntask ? (ntask - 1 - t0) / G + 1 : 0;
    const uint32_t* fw = reinterpret_cast<const uint32_t*>(fb);
    const uint32_t* gw = reinterpret_cast<const uint32_t*>(gb);
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], ring_arrivals(sg.items, kConsumerWarps));
        }
        mbar_init_fence();
    }
    pdl_wait();
    __syncthreads();

    if (warp == kConsumerWarps) {  // producer: lane k < 19 fetches slot k
        const int k = lane < kSlots ? lane : 0;
        const int a = dir_of(k), ex = ex9(a), ey = ey9(a);
        const uint32_t* base = k < 9 ? fw : gw;
        const uint32_t* bn = base + (int64_t)plane_of(k, a) * NP;
        const uint32_t* bw = base + (int64_t)plane_of(k, opp9(a)) * NP;
        int64_t it = 0;
        for (; it < nmine; ++it) {
            const int s = (int)(it % kStages);
            const int64_t u = it / kStages;
            if (u > 0 && !mbar_wait_bounded(&empty[s], (uint32_t)(u - 1) & 1u, kWaitNs)) {
                if (lane == 0) atomicExch(err, 1);
                break;
            }
            const int64_t t = t0 + it * G;
            const int y = (int)(t / nseg), w0 = (int)(t % nseg) * segw;
            const int TW = min(segw, H - w0);
            const bool wall = (ey == 1 && y == 0) || (ey == -1 && y == ny - 1);
            uint32_t* dst = stage0 + s * kStageW + k * kSlotW;
            // this lane's copies: (global word offset, shared word offset, words)
            int64_t g0 = 0, g1 = 0, g2 = 0;
            int d0 = 0, d1 = 0, d2 = 0, n0 = 0, n1 = 0, n2 = 0;
            if (lane < kSlots) {
                if (wall) {
                    if (CLOSURE == 0) g0 = (int64_t)y * H + w0, d0 = kHaloW, n0 = TW;
                } else {
                    const int64_t row = (int64_t)(y - ey) * H;
                    if (ex == 0) {
                        g0 = row + w0, d0 = kHaloW, n0 = TW;
                    } else if (w0 >= kHaloW && w0 + TW + kHaloW <= H) {  // both halos in one copy
                        g0 = row + w0 - kHaloW, d0 = 0, n0 = TW + 2 * kHaloW;
                    } else {
                        g0 = row + w0, d0 = kHaloW, n0 = TW;
                        if (ex == 1) g1 = row + (w0 == 0 ? H - kHaloW : w0 - kHaloW), d1 = 0, n1 = kHaloW;
                        else g2 = row + (w0 + TW == H ? 0 : w0 + TW), d2 = kHaloW + TW, n2 = kHaloW;
                    }
                }
            }
            const uint32_t mine = 4u * (uint32_t)(n0 + n1 + n2);
            const uint32_t bytes = __reduce_add_sync(0xffffffffu, mine);
            if (lane == 0) mbar_arrive_expect_tx(&full[s], bytes);
            __syncwarp();
            const uint32_t* src = (wall && CLOSURE == 0) ? bw : bn;
            if (n0) bulk_g2s(dst + d0, src + g0, 4u * n0, &full[s]);
            if (n1) bulk_g2s(dst + d1, src + g1, 4u * n1, &full[s]);
            if (n2) bulk_g2s(dst + d2, src + g2, 4u * n2, &full[s]);
        }
        for (int s = 0; s < kStages; ++s) {
            if (it <= s) continue;
            const int64_t u_last = (it - 1 - s) / kStages;
            if (!mbar_wait_bounded(&full[s], (uint32_t)u_last & 1u, kWaitNs) && lane == 0) atomicExch(err, 1);
        }
        return;
    }

    typedef Packed<S> P;
    const int dy = (int)(G / nseg), dg = (int)(G % nseg);
    const auto skip = [&](uint32_t it) -> bool { return pass_task(full, empty, it, lane, err); };
    ItemWalk<kConsumerWarps> i(warp);
    TaskAt at(nseg);
    for (; i.next((uint32_t)nmine, sg.items, skip); i.c += kConsumerWarps) {
        at.to(i.it, nseg, dy, dg);
        const uint32_t s = i.it % kStages;
        if (!mbar_wait_bounded(&full[s], (i.it / kStages) & 1u, kWaitNs)) {
            atomicExch(err, 1);
            break;
        }
        const int y = at.y, w = at.g * segw + 32 * i.c + lane;  // the lane's word in its row
        const bool active = w < H;
        {
            const bool bottom = (y == 0), top = (y == ny - 1);
            const uint32_t* st = stage0 + s * kStageW + kHaloW + 32 * i.c + lane;
            const bool sm = (w == 0), sp = (w == H - 1);      // halves swap across the row edge
            const int wm = sm ? H - 1 : w - 1, wp = sp ? 0 : w + 1;
            auto body = [&](auto walls) {
                constexpr bool W = decltype(walls)::value;
                uint32_t u[kSlots];
                if (active) {
#pragma unroll
                    for (int k = 0; k < kSlots; ++k) {
                        const int a = dir_of(k), ex = ex9(a), ey = ey9(a);
                        const bool wall = W && ((ey == 1 && bottom) || (ey == -1 && top));
                        const uint32_t* row = st + k * kSlotW;
                        if (wall || ex == 0)
                            u[k] = row[0];
                        else if (ex == 1)  // nodes x - 1: the word before (swapped across the left edge)
                            u[k] = sm ? __byte_perm(row[-1], 0, 0x1032) : row[-1];
                        else  // nodes x + 1: the word after (swapped across the right edge)
                            u[k] = sp ? __byte_perm(row[1], 0, 0x1032) : row[1];
                    }
                }
                // release the stage at once, as the two-buffer kernel does
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[s]);
                if (!active) return;
                float2 v[kSlots];
#pragma unroll
                for (int k = 0; k < kSlots; ++k) v[k] = P::pair(u[k]);
                float2 f[9], gx[5], gy[5];
#pragma unroll
                for (int a = 0; a < 9; ++a) f[a] = v[a];
#pragma unroll
                for (int a = 0; a < 5; ++a) {
                    gx[a] = v[9 + a];
                    gy[a] = v[14 + a];
                }
                if (W && CLOSURE == 0) {
                    if (bottom) {
                        const WallCoef<float>& wc = p.bot;
                        f[5] = f[5] + wc.du;
                        f[6] = f[6] - wc.du;
                        gx[2] = ffma(wc.r, gx[2], wc.kx);
                        gy[2] = -gy[2];
                    }
                    if (top) {
                        const WallCoef<float>& wc = p.top;
                        f[7] = f[7] - wc.du;
                        f[8] = f[8] + wc.du;
                        gx[4] = ffma(wc.r, gx[4], wc.kx);
                        gy[4] = -gy[4];
                    }
                }
                close_collide_pair<CLOSURE, COUPLING, W>(f, gx, gy, p, bottom, top);
                // push: direction b -> plane bbar at x + e_b; through a wall -> plane b, own word
                const uint32_t rc = (uint32_t)y * H, rs = rc - H, rn = rc + H;
                auto put = [&](int k, uint32_t at, bool swap, float2 q) {
                    put_word(out, k, 4u * at, swap ? P::pack(q.y, q.x) : P::pack(q.x, q.y));
                };
                put(0, rc + w, false, f[0]);
                put(3, rc + wp, sp, f[1]);
                put(1, rc + wm, sm, f[3]);
                put(9, rc + w, false, gx[0]);
                put(12, rc + wp, sp, gx[1]);
                put(10, rc + wm, sm, gx[3]);
                put(14, rc + w, false, gy[0]);
                put(17, rc + wp, sp, gy[1]);
                put(15, rc + wm, sm, gy[3]);
                if (!top) {
                    put(4, rn + w, false, f[2]);
                    put(7, rn + wp, sp, f[5]);
                    put(8, rn + wm, sm, f[6]);
                    put(13, rn + w, false, gx[2]);
                    put(18, rn + w, false, gy[2]);
                } else {
                    put(2, rc + w, false, f[2]);
                    put(5, rc + w, false, f[5]);
                    put(6, rc + w, false, f[6]);
                    put(11, rc + w, false, gx[2]);
                    put(16, rc + w, false, gy[2]);
                }
                if (!bottom) {
                    put(2, rs + w, false, f[4]);
                    put(5, rs + wm, sm, f[7]);
                    put(6, rs + wp, sp, f[8]);
                    put(11, rs + w, false, gx[4]);
                    put(16, rs + w, false, gy[4]);
                } else {
                    put(4, rc + w, false, f[4]);
                    put(7, rc + w, false, f[7]);
                    put(8, rc + w, false, f[8]);
                    put(13, rc + w, false, gx[4]);
                    put(18, rc + w, false, gy[4]);
                }
            };
            if (bottom || top)
                body(std::true_type{});
            else
                body(std::false_type{});
        }
    }
}

// Failure detection without a GPU fault: one warp waits, with the staged kernels' bounded wait, on
// a freshly initialised mbarrier that nothing arrives on (its first phase never completes), gives
// up after limit_ns and records the timeout in *err as a staged step's wait would.  No copy is in
// flight to that barrier, so returning is safe.
__global__ void wait_timeout_probe_kernel(int* err, uint64_t limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_init_fence();
    }
    __syncwarp();
    if (threadIdx.x == 0 && !mbar_wait_bounded(&bar, 0, limit_ns)) atomicExch(err, 1);
}

template <typename K>
cudaError_t prepare_kernel(K kernel, int* blocks, size_t smem = kSmem) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kThreads, smem);
    if (e == cudaSuccess && occ < 1) e = cudaErrorInvalidConfiguration;
    *blocks = occ;
    return e;
}

// Every closure / coupling instance of the two-buffer kernel (inplace = 0) or of the in-place
// phase-0 kernel (inplace = 1); *blocks = the smallest number resident per SM.
template <typename S>
cudaError_t prepare_typed(int inplace, int* blocks) {
    int b[4] = {0, 0, 0, 0};
    cudaError_t e;
    if (inplace) {
        e = prepare_kernel(step_kernel_aa_staged<S, 0, 0>, &b[0], kSmem);
        if (e == cudaSuccess) e = prepare_kernel(step_kernel_aa_staged<S, 1, 0>, &b[1], kSmem);
        if (e == cudaSuccess) e = prepare_kernel(step_kernel_aa_staged<S, 0, 1>, &b[2], kSmem);
        if (e == cudaSuccess) e = prepare_kernel(step_kernel_aa_staged<S, 1, 1>, &b[3], kSmem);
    } else {
        e = prepare_kernel(step_kernel_staged<S, 0, 0>, &b[0], kSmem);
        if (e == cudaSuccess) e = prepare_kernel(step_kernel_staged<S, 1, 0>, &b[1], kSmem);
        if (e == cudaSuccess) e = prepare_kernel(step_kernel_staged<S, 0, 1>, &b[2], kSmem);
        if (e == cudaSuccess) e = prepare_kernel(step_kernel_staged<S, 1, 1>, &b[3], kSmem);
    }
    *blocks = std::min(std::min(b[0], b[1]), std::min(b[2], b[3]));
    return e;
}

template <typename S>
SlotPlanes planes_of(S* f, S* g, int64_t N) {
    SlotPlanes d;
    for (int k = 0; k < kSlots; ++k) d.slot[k] = k < 9 ? f + k * N : g + (k - 9) * N;
    return d;
}

template <typename S>
void launch_typed_aa_staged(void* f, void* g, const StepParams<float>& p, int closure, const StagedStep& ss,
                            cudaStream_t st) {
    const Segments sg = segments_of(p.nx);
    const unsigned grid = (unsigned)std::min<int64_t>((int64_t)p.ny * sg.n, ss.grid);
    S* fb = (S*)f;
    S* gb = (S*)g;
    const auto kernel = p.coupling == 0
                            ? (closure == 0 ? step_kernel_aa_staged<S, 0, 0> : step_kernel_aa_staged<S, 1, 0>)
                            : (closure == 0 ? step_kernel_aa_staged<S, 0, 1> : step_kernel_aa_staged<S, 1, 1>);
    launch_pdl(kernel, grid, kThreads, kSmem, st, (const S*)fb, (const S*)gb, planes_of(fb, gb, p.N), p, sg, ss.err);
}

template <typename S>
void launch_typed_staged(const void* fin, const void* gin, void* fout, void* gout, const StepParams<float>& p,
                         int closure, const StagedStep& ss, cudaStream_t st) {
    const Segments sg = segments_of(p.nx);
    const unsigned grid = (unsigned)std::min<int64_t>((int64_t)p.ny * sg.n, ss.grid);
    const auto kernel = p.coupling == 0 ? (closure == 0 ? step_kernel_staged<S, 0, 0> : step_kernel_staged<S, 1, 0>)
                                        : (closure == 0 ? step_kernel_staged<S, 0, 1> : step_kernel_staged<S, 1, 1>);
    launch_pdl(kernel, grid, kThreads, kSmem, st, (const S*)fin, (const S*)gin, planes_of((S*)fout, (S*)gout, p.N), p,
               sg, ss.err);
}

}  // namespace

bool staged_step_applies(int storage, int nx, int inplace) {
    (void)inplace;  // two buffers: the whole step; in place: phase 0 of each pair
    return storage >= 2 && nx % 8 == 0 && nx >= kSegX;
}

cudaError_t prepare_staged_step(int storage, int inplace, unsigned* grid) {
    int dev = 0, sms = 0, blocks = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = storage == 2 ? prepare_typed<__nv_bfloat16>(inplace, &blocks) : prepare_typed<__half>(inplace, &blocks);
    *grid = (unsigned)(sms * blocks);
    return e;
}

cudaError_t launch_wait_timeout_probe(int* err, uint64_t limit_ns, cudaStream_t st) {
    wait_timeout_probe_kernel<<<1, 32, 0, st>>>(err, limit_ns);
    return cudaGetLastError();
}

cudaError_t launch_step_aa_staged(int storage, int closure, void* f, void* g, const StepParams<float>& p,
                                  const StagedStep& ss, cudaStream_t st) {
    if (storage == 2)
        launch_typed_aa_staged<__nv_bfloat16>(f, g, p, closure, ss, st);
    else
        launch_typed_aa_staged<__half>(f, g, p, closure, ss, st);
    return cudaGetLastError();
}

cudaError_t launch_step_staged(int storage, int closure, const void* fin, const void* gin, void* fout, void* gout,
                               const StepParams<float>& p, const StagedStep& ss, cudaStream_t st) {
    if (storage == 2)
        launch_typed_staged<__nv_bfloat16>(fin, gin, fout, gout, p, closure, ss, st);
    else
        launch_typed_staged<__half>(fin, gin, fout, gout, p, closure, ss, st);
    return cudaGetLastError();
}

}  // namespace lks
