// lks_resident.cuh -- a lattice held in the shared memory of one thread-block cluster for as many steps as a
// call asks for.
//
// A small lattice's step is launch and memory latency: in a graph of single-step kernels a 4 x 65 channel
// took 1.7 us a step in FP32 and a 4 x 257 one 2.2; here they take 0.79 and 0.74 (64 x 64: 1.41 -> 0.88).
// The CTAs of a cluster hold a band of rows each, in two buffers (a step reads one and writes the other);
// after a step each CTA stores the populations that leave its band into the halo rows of the neighbouring
// bands (distributed shared memory), and one cluster barrier, 0.2 us at any cluster size up to 16, ends the
// step.  A CTA that is one barrier ahead writes halo rows of the buffer its neighbour is not reading.  The
// per-node operations are the ordinary step's, so are the bits.
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
};

// One step of a band, one node per thread and pass: buffer b -> buffer b ^ 1.  The caller ends the step
// with a cluster barrier.  The pulls and link closures of step_node_with in 32-bit indices.
template <typename S, typename C, int CLOSURE, int COUPLING>
__device__ __forceinline__ void band_step(const Band<S>& band, int b, const StepParams<C>& p) {
    typedef Loader<S, C, false> L;
    const int nx = band.nx, P = band.plane;
    for (int i = band.i0, jl = band.j0; jl < band.rows; i += band.di, jl += band.dj) {
        if (i >= nx) {
            i -= nx;
            if (++jl >= band.rows) break;
        }
        const int j = band.first + jl;
        const bool bottom = j == 0, top = j == p.ny - 1;
        const int n = (jl + 1) * nx + i;
        const int l = i == 0 ? nx - 1 : -1, r = i == nx - 1 ? 1 - nx : 1;  // to the left and right column
        const S* c = band.buf(b) + n;
        C f[9], gx[5], gy[5];
        f[0] = L::ld(c);
        f[1] = L::ld(c + 1 * P + l);
        f[3] = L::ld(c + 3 * P + r);
        gx[0] = L::ld(c + 9 * P);
        gx[1] = L::ld(c + 10 * P + l);
        gx[3] = L::ld(c + 12 * P + r);
        gy[0] = L::ld(c + 14 * P);
        gy[1] = L::ld(c + 15 * P + l);
        gy[3] = L::ld(c + 17 * P + r);
        if (!bottom) {
            const S* s = c - nx;
            f[2] = L::ld(s + 2 * P);
            f[5] = L::ld(s + 5 * P + l);
            f[6] = L::ld(s + 6 * P + r);
            gx[2] = L::ld(s + 11 * P);
            gy[2] = L::ld(s + 16 * P);
        } else if (CLOSURE == 0) {
            f[2] = L::ld(c + 4 * P);
            f[5] = L::ld(c + 7 * P) + p.bot.du;
            f[6] = L::ld(c + 8 * P) - p.bot.du;
            gx[2] = ffma(p.bot.r, L::ld(c + 13 * P), p.bot.kx);
            gy[2] = -L::ld(c + 18 * P);
        }
        if (!top) {
            const S* s = c + nx;
            f[4] = L::ld(s + 4 * P);
            f[7] = L::ld(s + 7 * P + r);
            f[8] = L::ld(s + 8 * P + l);
            gx[4] = L::ld(s + 13 * P);
            gy[4] = L::ld(s + 18 * P);
        } else if (CLOSURE == 0) {
            f[4] = L::ld(c + 2 * P);
            f[7] = L::ld(c + 5 * P) - p.top.du;
            f[8] = L::ld(c + 6 * P) + p.top.du;
            gx[4] = ffma(p.top.r, L::ld(c + 11 * P), p.top.kx);
            gy[4] = -L::ld(c + 16 * P);
        }
        if (CLOSURE == 1) {
            if (bottom) moment_closure_bottom<C, COUPLING>(f, gx, gy, p.bot, p);
            if (top) moment_closure_top<C, COUPLING>(f, gx, gy, p.top, p);
        }
        collide<C, COUPLING>(f, gx, gy, p);
        S* o = band.buf(b ^ 1) + n;
#pragma unroll
        for (int a = 0; a < 9; ++a) store_s<S, C>(o + a * P, f[a]);
#pragma unroll
        for (int a = 0; a < 5; ++a) store_s<S, C>(o + (9 + a) * P, gx[a]);
#pragma unroll
        for (int a = 0; a < 5; ++a) store_s<S, C>(o + (14 + a) * P, gy[a]);
        // populations that leave the band, into the neighbours' halo rows
        const int half = (b ^ 1) * (19 * P);
        if (jl == 0 && band.below) {
            S* t = band.below + half + (band.rows_below + 1) * nx + i;
            store_s<S, C>(t + 4 * P, f[4]);
            store_s<S, C>(t + 7 * P, f[7]);
            store_s<S, C>(t + 8 * P, f[8]);
            store_s<S, C>(t + 13 * P, gx[4]);
            store_s<S, C>(t + 18 * P, gy[4]);
        }
        if (jl == band.rows - 1 && band.above) {
            S* t = band.above + half + i;
            store_s<S, C>(t + 2 * P, f[2]);
            store_s<S, C>(t + 5 * P, f[5]);
            store_s<S, C>(t + 6 * P, f[6]);
            store_s<S, C>(t + 11 * P, gx[2]);
            store_s<S, C>(t + 16 * P, gy[2]);
        }
    }
}

}  // namespace lks
