// lks_resident.cu -- lks_step of small lattices: n steps in one launch of one cluster (lks_resident.cuh).
#include <algorithm>

#include "lks_internal.h"
#include "lks_quad.cuh"
#include "lks_resident.cuh"

namespace lks {
namespace {

constexpr size_t kResidentSmem = 200 * 1024;  // most dynamic shared memory of a CTA

template <typename S, typename C, int CLOSURE, int COUPLING>
__global__ void __launch_bounds__(sizeof(C) == 8 ? kResidentThreads / 2 : kResidentThreads)
    resident_kernel(const S* fin, const S* gin, S* fout, S* gout, const StepParams<C> p, int rows_max, int ilv,
                    int steps) {
    extern __shared__ __align__(16) unsigned char res_sm[];
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    Band<S> band;
    band.set(reinterpret_cast<S*>(res_sm), p.nx, p.ny, rows_max);
    band.load(fin, gin, p.N, p.ny, ilv);
    cl.sync();  // every band is loaded before anyone stores, and every CTA runs before its memory is written
    int b = 0;
    for (int s = 0; s < steps; ++s, b ^= 1) {
        band_step<S, C, CLOSURE, COUPLING>(band, b, p);
        cl.sync();
    }
    band.store(b, fout, gout, p.N, ilv);
}

// FP64, at most 32 nodes a CTA and group: four warps to a group (lks_quad.cuh).
template <int CLOSURE>
__global__ void __launch_bounds__(128 * kResidentQuads) resident_quad_kernel(const double* fin, const double* gin,
                                                                             double* fout, double* gout,
                                                                             const StepParams<double> p, int rows_max,
                                                                             int ilv, int steps) {
    extern __shared__ __align__(16) unsigned char res_sm[];
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    Band<double> band;
    band.set(reinterpret_cast<double*>(res_sm), p.nx, p.ny, rows_max);
    band.load(fin, gin, p.N, p.ny, ilv);
    double* sh = reinterpret_cast<double*>(res_sm) + 2 * 19 * band.plane;
    cl.sync();
    int b = 0;
    for (int s = 0; s < steps; ++s, b ^= 1) {
        if (p.Fx != 0.0)
            quad_step<CLOSURE, true>(band, b, p, sh);
        else
            quad_step<CLOSURE, false>(band, b, p, sh);
        cl.sync();
    }
    band.store(b, fout, gout, p.N, ilv);
}

template <typename S, typename C>
struct Resident {
    typedef void (*Fn)(const S*, const S*, S*, S*, const StepParams<C>, int, int, int);
    static Fn kernel(int closure, int coupling, bool quads) {
        if constexpr (sizeof(C) == 8)
            if (quads) return closure == 0 ? resident_quad_kernel<0> : resident_quad_kernel<1>;
        if (coupling == 0) return closure == 0 ? resident_kernel<S, C, 0, 0> : resident_kernel<S, C, 1, 0>;
        return closure == 0 ? resident_kernel<S, C, 0, 1> : resident_kernel<S, C, 1, 1>;
    }
    static void config(cudaLaunchConfig_t* lc, cudaLaunchAttribute* at, const ResidentPlan& rp, cudaStream_t st) {
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim.x = rp.ctas;
        at->val.clusterDim.y = at->val.clusterDim.z = 1;
        lc->gridDim = dim3(rp.ctas);
        lc->blockDim = dim3(rp.threads);
        lc->dynamicSmemBytes = rp.smem;
        lc->stream = st;
        lc->attrs = at;
        lc->numAttrs = 1;
    }
    // rp.ctas = 0 if no cluster of that size and shared memory can run.
    static cudaError_t prepare(int closure, int coupling, ResidentPlan* rp) {
        Fn k = kernel(closure, coupling, rp->quads > 0);
        cudaLaunchConfig_t lc = {};
        cudaLaunchAttribute at[1];
        int clusters = 0;
        // the limit is the function's, shared by every handle: always the same value
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResidentSmem);
        if (e == cudaSuccess && rp->ctas > 8)
            e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess) {
            config(&lc, at, *rp, nullptr);
            e = cudaOccupancyMaxActiveClusters(&clusters, k, &lc);
        }
        if (e != cudaSuccess || clusters < 1) {
            cudaGetLastError();
            rp->ctas = 0;
        }
        return cudaSuccess;
    }
    static cudaError_t launch(const void* fin, const void* gin, void* fout, void* gout, const StepParams<C>& p,
                              int closure, const ResidentPlan& rp, int ilv, int steps, cudaStream_t st) {
        cudaLaunchConfig_t lc = {};
        cudaLaunchAttribute at[1];
        config(&lc, at, rp, st);
        return cudaLaunchKernelEx(&lc, kernel(closure, p.coupling, rp.quads > 0), (const S*)fin, (const S*)gin,
                                  (S*)fout, (S*)gout, p, rp.rows_max, ilv, steps);
    }
};

}  // namespace

cudaError_t plan_resident(int storage, int closure, int coupling, int nx, int ny, ResidentPlan* rp) {
    *rp = ResidentPlan{};
    const int64_t N = (int64_t)nx * ny;
    if (N > (storage == 0 ? kResidentNodesF64 : (storage == 1 ? kResidentNodesF32 : kResidentNodes16)))
        return cudaSuccess;
    int ctas = N <= 512 && storage != 0 ? 8 : 16;
    while (ctas > ny) ctas /= 2;
    rp->rows_max = (ny + ctas - 1) / ctas;
    const int nodes = rp->rows_max * nx;
    if (storage == 0 && nodes > kResidentCtaNodesF64) return cudaSuccess;
    rp->threads = std::min(storage == 0 ? kResidentThreads / 2 : kResidentThreads, (nodes + 31) / 32 * 32);
    rp->smem = (size_t)2 * 19 * nx * (rp->rows_max + 2) * storage_bytes(storage);
    if (storage == 0 && coupling == 0 && nodes <= 32 * kResidentQuads) {
        rp->quads = (nodes + 31) / 32;
        rp->threads = 128 * rp->quads;
        rp->smem += rp->quads * kQuadWords * sizeof(double);
    }
    if (rp->smem > kResidentSmem) return cudaSuccess;
    rp->ctas = ctas;
    rp->least = resident_least(storage, N);
    switch (storage) {
        case 0: return Resident<double, double>::prepare(closure, coupling, rp);
        case 1: return Resident<float, float>::prepare(closure, coupling, rp);
        case 2: return Resident<__nv_bfloat16, float>::prepare(closure, coupling, rp);
        default: return Resident<__half, float>::prepare(closure, coupling, rp);
    }
}

cudaError_t launch_resident(int storage, int closure, const void* fin, const void* gin, void* fout, void* gout,
                            const StepParams<double>& pd, const ResidentPlan& rp, int ilv, int steps, cudaStream_t st) {
    if (storage == 0) return Resident<double, double>::launch(fin, gin, fout, gout, pd, closure, rp, ilv, steps, st);
    const StepParams<float> p = convert_params<float>(pd);
    if (storage == 1) return Resident<float, float>::launch(fin, gin, fout, gout, p, closure, rp, ilv, steps, st);
    if (storage == 2)
        return Resident<__nv_bfloat16, float>::launch(fin, gin, fout, gout, p, closure, rp, ilv, steps, st);
    return Resident<__half, float>::launch(fin, gin, fout, gout, p, closure, rp, ilv, steps, st);
}

}  // namespace lks
