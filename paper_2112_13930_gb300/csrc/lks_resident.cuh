// lks_resident.cuh -- a lattice held in the shared memory of one thread-block cluster for as many steps as a
// call asks for.
//
// A small lattice's step is launch and memory latency: in a graph of single-step kernels a 4 x 65 channel
// took 1.7 us a step in FP32 and a 4 x 257 one 2.2; here they take 0.79 and 0.74 (64 x 64: 1.41 -> 0.88).  Here the CTAs of a cluster hold a band of rows each, in two buffers (a step
// reads one and writes the other); after a step each CTA stores the populations that leave its band into the
// halo rows of the neighbouring bands (distributed shared memory), and one cluster barrier, 0.2 us at any
// cluster size up to 16, ends the step.  A CTA that is one barrier ahead writes halo rows of the buffer its
// neighbour is not reading.  The per-node step is the ordinary one, so are the bits.
#pragma once
#include <cooperative_groups.h>

#include "lks_device.cuh"

namespace lks {

// Rows [first, first + rows) of the lattice in this CTA, with a halo row below (local row 0) and above.
template <typename S>
struct Band {
    S* base;        // two buffers of [19][rows_max + 2][nx]: f0..8, gx0..4, gy0..4
    int nx, first, rows;
    int plane;      // nx (rows_max + 2)
    S* below;       // the neighbouring bands' buffers; null at a wall
    S* above;
    int rows_below;
    int i0, j0, di, dj;  // this thread's first node and the stride between its nodes, in columns and rows

    __device__ static int first_of(int rank, int cs, int ny) { return (int)((int64_t)ny * rank / cs); }
    __device__ __forceinline__ S* buf(int b) const { return base + b * (19 * plane); }

    // `sm`: this CTA's shared memory, the same offset in every CTA of the cluster.
    __device__ void set(S* sm, int nx_, int ny, int rows_max) {
        cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
        const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
        nx = nx_;
        first = first_of(rank, cs, ny);
        rows = first_of(rank + 1, cs, ny) - first;
        rows_below = rank > 0 ? first - first_of(rank - 1, cs, ny) : 0;
        plane = nx * (rows_max + 2);
        base = sm;
        j0 = (int)threadIdx.x / nx;
        i0 = (int)threadIdx.x - j0 * nx;
        dj = (int)blockDim.x / nx;
        di = (int)blockDim.x - dj * nx;
        below = rank > 0 ? cl.map_shared_rank(sm, rank - 1) : nullptr;
        above = rank + 1 < cs ? cl.map_shared_rank(sm, rank + 1) : nullptr;
    }

    // Global state -> buffer 0, the halo rows included (they are other bands' rows).  ilv: row length if the
    // stored rows are interleaved (in-place 16-bit handles), else 0.
    __device__ void load(const S* f, const S* g, int64_t N, int ny, int ilv) {
        const int lo = first > 0 ? -1 : 0, hi = first + rows < ny ? rows + 1 : rows;
        const int count = (hi - lo) * nx;
        for (int a = 0; a < 19; ++a) {
            const S* src = a < 9 ? f + a * N : g + (a - 9) * N;
            for (int k = threadIdx.x; k < count; k += blockDim.x) {
                const int j = k / nx + lo, i = k - (k / nx) * nx;
                base[a * plane + (j + 1) * nx + i] = src[slot(first + j, i, ilv)];
            }
        }
    }
    // Buffer b -> global state (the band's own rows).
    __device__ void store(int b, S* f, S* g, int64_t N, int ilv) const {
        for (int a = 0; a < 19; ++a) {
            S* dst = a < 9 ? f + a * N : g + (a - 9) * N;
            for (int k = threadIdx.x; k < rows * nx; k += blockDim.x) {
                const int j = k / nx, i = k - j * nx;
                dst[slot(first + j, i, ilv)] = buf(b)[a * plane + (j + 1) * nx + i];
            }
        }
    }
    __device__ int64_t slot(int y, int x, int ilv) const {
        const int h = nx >> 1;
        return (int64_t)y * nx + (ilv == 0 ? x : (x < h ? 2 * x : 2 * (x - h) + 1));
    }

    // Populations of local row j (of buffer b) that leave the band, into the neighbours' halo rows.
    __device__ __forceinline__ void hand_over(int b, int i, int j) const {
        const S* own = buf(b) + (j + 1) * nx + i;
        const int dn[5] = {4, 7, 8, 9 + 4, 14 + 4}, up[5] = {2, 5, 6, 9 + 2, 14 + 2};
        if (j == 0 && below) {
            S* to = below + b * (19 * plane) + (rows_below + 1) * nx + i;
#pragma unroll
            for (int q = 0; q < 5; ++q) to[dn[q] * plane] = own[dn[q] * plane];
        }
        if (j == rows - 1 && above) {
            S* to = above + b * (19 * plane) + i;
#pragma unroll
            for (int q = 0; q < 5; ++q) to[up[q] * plane] = own[up[q] * plane];
        }
    }
};

// One step of a band, one node per thread and pass: buffer b -> buffer b ^ 1.  q: the lattice's parameters
// with N = band.plane.  The caller ends the step with a cluster barrier.
template <typename S, typename C, int CLOSURE, int COUPLING>
__device__ __forceinline__ void band_step(const Band<S>& band, int b, const StepParams<C>& q) {
    const S* in = band.buf(b);
    S* out = band.buf(b ^ 1);
    for (int i = band.i0, j = band.j0; j < band.rows; i += band.di, j += band.dj) {
        if (i >= band.nx) {
            i -= band.nx;
            if (++j >= band.rows) break;
        }
        step_node_with<S, C, CLOSURE, Loader<S, C, false>, COUPLING>(in, in + 9 * band.plane, out, out + 9 * band.plane,
                                                                     q, (j + 1) * band.nx + i, i, band.first + j);
        band.hand_over(b ^ 1, i, j);
    }
}

}  // namespace lks
