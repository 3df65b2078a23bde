// lb_diffuse.cu -- the stress-diffusion sub-step kernel of one lattice (lb_diffuse.cuh) and its launcher.
#include <cuda_runtime.h>

#include "lb_cell.cuh"
#include "lb_diffuse.cuh"

namespace vlb {

using namespace dif;

int diffuse_tiles_x(int nx) { return (nx + DX - 1) / DX; }
int diffuse_tiles_y(int ny) { return (ny + DY - 1) / DY; }

namespace {

// One sub-step, started by programmatic dependent launch behind the lattice kernel or the sub-step
// before it (on a lattice of one wave of tiles a launch that waits for the end of the former one costs
// more than the sub-step: 333 x 190, three sub-steps, 42.2 -> 30.3 us per step).  early: the kernel behind
// this one waits for it before it reads anything.
__global__ void __launch_bounds__(DNT) k_diffuse(const float* src, float* dst, long long NP, int nx, int ny, float D, int early)
{
    extern __shared__ __align__(16) float sm[];
    cell::pdl_wait();
    if (early) cell::pdl_trigger();
    diffuse_steps<1>(src, dst, NP, nx, ny, D, blockIdx.x, blockIdx.y, sm);
}

__global__ void __launch_bounds__(256) k_copy3(const float* src, float* dst, long long NP, int early)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    cell::pdl_wait();
    if (early) cell::pdl_trigger();
    if (i < NP) {
        const float v[3] = {src[i], src[NP + i], src[2 * NP + i]};
        dst[i] = v[0];
        dst[NP + i] = v[1];
        dst[2 * NP + i] = v[2];
    }
}

}  // namespace

cudaError_t launch_diffusion(float* sig_new, float* sig_tmp, long long NP, int nx, int ny, float D, int substeps,
                             cudaStream_t s, bool pdl, bool next_waits)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(diffuse_tiles_x(nx), diffuse_tiles_y(ny));
    cfg.blockDim = dim3(DNT);
    cfg.dynamicSmemBytes = sizeof(float) * steps_smem(1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    const int n = substeps + (substeps & 1);      // an odd number ends in the other buffer: copied back
    for (int k = 0; k < n; ++k) {
        const float* src = (k & 1) ? sig_tmp : sig_new;
        float* dst = (k & 1) ? sig_new : sig_tmp;
        const int early = k + 1 < n || next_waits;
        cudaError_t e;
        if (k < substeps) {
            e = cudaLaunchKernelEx(&cfg, k_diffuse, src, dst, NP, nx, ny, D, early);
        } else {
            cfg.gridDim = dim3((unsigned)((NP + 255) / 256));
            cfg.blockDim = dim3(256);
            cfg.dynamicSmemBytes = 0;
            e = cudaLaunchKernelEx(&cfg, k_copy3, src, dst, NP, early);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace vlb
