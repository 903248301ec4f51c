// lks_ring.cuh -- how the consumer warps of a staged kernel share the items of their block's tasks.
//
// A producer stages task after task in a ring of shared-memory stages, each with a `full` and an `empty`
// mbarrier.  Warp w of WARPS consumer warps takes items w, w + WARPS, ... of the stream of all tasks' items, so
// with fewer items than warps it has none in some tasks.  An mbarrier wait names a phase by its parity and so can
// tell only the current phase from the one before, and copies into different stages may land in any order: a warp
// that went past a task without waiting for its copies could take that phase, still open, for the completed one of
// the same parity two phases on.  Therefore every warp waits for every task, in order, and arrives on every task's
// `empty`: once per item, after reading it, or once where it has none.  A phase of `empty` then ends only when each
// warp has seen the task's copies, a phase of `full` begins only after that, and no barrier is ever more than the
// one phase ahead that its waiters can tell.  Plain C++, so that a host program can enumerate it.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define LKS_RING_FN __host__ __device__ __forceinline__
#else
#define LKS_RING_FN inline
#endif

namespace lks {

// Arrivals that end a phase of `empty`: one per item (a warp with two items arrives twice), and one from each warp
// without an item; WARPS consecutive items belong to as many warps.
LKS_RING_FN constexpr int ring_arrivals(int items, int warps) { return items > warps ? items : warps; }

template <int WARPS>
struct ItemWalk {
    uint32_t it;  // task of the block
    int c;        // item of the task
    LKS_RING_FN explicit ItemWalk(int warp) : it(0), c(warp) {}
    // The item at or after (it, c); false: no more.  skip(it) has to wait for task it, in which the warp has no
    // item, and to arrive; false from it ends the walk.  After an item: c += WARPS.
    template <typename Skip>
    LKS_RING_FN bool next(uint32_t ntask, int items, Skip skip) {
        while (c >= items) {
            // c >= WARPS: the warp's last item was in this task
            if (c < WARPS && it < ntask && !skip(it)) return false;
            c -= items;
            ++it;
        }
        return it < ntask;
    }
};

}  // namespace lks
