// lks_pair.cuh -- moment closure and collision of two nodes held as float2 values, for the kernels
// that take two nodes per thread.
#pragma once
#include "lks_device.cuh"

namespace lks {

// Moment closure (wall rows, W) and collision of a node pair.  The Maxwell coupling runs as one
// float2.  The Lorentz coupling runs per node in scalar, as the one- and two-node kernels do: on its
// f update the scalar and the packed forms were measured to round differently in a fraction of the
// nodes, which would end the agreement bit for bit between the kernels.
template <int CLOSURE, int COUPLING, bool W>
__device__ __forceinline__ void close_collide_pair(float2 f[9], float2 gx[5], float2 gy[5], const StepParams<float>& p,
                                                   bool bottom, bool top) {
    if constexpr (COUPLING == 0) {
        if (W && CLOSURE == 1) {
            if (bottom) moment_closure_bottom<float, 0>(f, gx, gy, p.bot, p);
            if (top) moment_closure_top<float, 0>(f, gx, gy, p.top, p);
        }
        collide<float, 0>(f, gx, gy, p);
    } else {
        float fA[9], gxA[5], gyA[5], fB[9], gxB[5], gyB[5];
#pragma unroll
        for (int a = 0; a < 9; ++a) fA[a] = f[a].x, fB[a] = f[a].y;
#pragma unroll
        for (int a = 0; a < 5; ++a) {
            gxA[a] = gx[a].x, gxB[a] = gx[a].y;
            gyA[a] = gy[a].x, gyB[a] = gy[a].y;
        }
        if (W && CLOSURE == 1) {
            if (bottom) {
                moment_closure_bottom<float, 1>(fA, gxA, gyA, p.bot, p);
                moment_closure_bottom<float, 1>(fB, gxB, gyB, p.bot, p);
            }
            if (top) {
                moment_closure_top<float, 1>(fA, gxA, gyA, p.top, p);
                moment_closure_top<float, 1>(fB, gxB, gyB, p.top, p);
            }
        }
        collide<float, 1>(fA, gxA, gyA, p);
        collide<float, 1>(fB, gxB, gyB, p);
#pragma unroll
        for (int a = 0; a < 9; ++a) f[a] = make_float2(fA[a], fB[a]);
#pragma unroll
        for (int a = 0; a < 5; ++a) {
            gx[a] = make_float2(gxA[a], gxB[a]);
            gy[a] = make_float2(gyA[a], gyB[a]);
        }
    }
}

}  // namespace lks
