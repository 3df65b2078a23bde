// lb_diffuse.cuh -- explicit stress-diffusion sub-steps for D_p beyond the Heun bound (device
// code shared by the diffusion kernel and the batched persistent kernel).
//
// Heun with the 5-point Laplacian is stable for 8 D_p <= 2.  For larger D_p the step takes the
// polymer-stress update of Eq. StiffCons without its diffusion term and then applies s Heun
// sub-steps of d sigma / dt = (D_p / s) lap sigma (periodic), each
//   sigma* = sigma + (D_p/s) lap sigma,  sigma' = sigma + (D_p/s) (lap sigma + lap sigma*) / 2.
// A pass of the batched form takes up to DMAX sub-steps at once: a tile stages sigma with a halo of two
// cells per sub-step and forms predictor and corrector in shared memory on a region that shrinks by
// a cell with each, so the sub-steps cost one launch and one trip through L2 instead of one each.
// Bound by latency (a launch's work on a lattice of one wave of tiles is 2 us): 20 lattices of
// 128^2 to 512^2, up to five sub-steps, 30 steps: 6493 us with a launch per sub-step, 6109 us so.
// At three the staged region is 2.4 times the tile.  lb_step launches every
// sub-step by itself (lb_launches_per_step counts them), started early: lb_diffuse.cu.
#pragma once
#include <cuda_runtime.h>

#include "lb_internal.h"

namespace vlb {
namespace dif {

constexpr int DX = 32, DY = 16, DNT = 256;
constexpr int DMAX = 3;          // sub-steps of one pass
// shared memory of a pass of s sub-steps (floats): sigma and its predictor on the staged region
constexpr int steps_smem(int s) { return 2 * 3 * (DX + 4 * s) * (DY + 4 * s); }
constexpr int SMEM = steps_smem(DMAX);

// The passes of d sub-steps: an even number, so that the result lies where the step left sigma
// (d = 1: one pass and a copy); pass k takes pass_steps(d, k) of them.
__host__ __device__ constexpr int passes(int d) { return 2 * ((d + 2 * DMAX - 1) / (2 * DMAX)); }
__host__ __device__ constexpr int pass_steps(int d, int k) { return d / passes(d) + (k < d % passes(d) ? 1 : 0); }

__device__ __forceinline__ int wrapd(int i, int n)
{
    i %= n;
    return i < 0 ? i + n : i;
}

// One DX x DY tile of a pass of S sub-steps; sm: SMEM floats, DNT threads.  A thread keeps the
// staged cells it loaded (value and first Laplacian) in registers, so only neighbours are read
// from shared memory.  The values are those of S single passes, bit for bit: every cell of the
// shrinking region is formed from the same numbers in the same order.
template <int S>
__device__ __forceinline__ void diffuse_steps(const float* src, float* dst, long long NP, int nx, int ny,
                                              float D, int bx, int by, float* sm)
{
    constexpr int W = DX + 4 * S, H = DY + 4 * S, N = W * H, C = (N + DNT - 1) / DNT;
    float* sA = sm;               // sigma [3][N]
    float* sB = sm + 3 * N;       // predictor [3][N]
    const int x0 = bx * DX - 2 * S, y0 = by * DY - 2 * S;
    // a staged index lies within one period of the lattice when the lattice is at least a tile and
    // its halo wide: one conditional add or subtract wraps it; smaller lattices take the modulo
    const bool near = nx >= W && ny >= H;
    float v[C][3], l0[C][3];
    int edge[C];                  // cells to the rim of the staged region (-1: no cell)
#pragma unroll
    for (int q = 0; q < C; ++q) {
        const int i = threadIdx.x + q * DNT;
        const int ly = i / W, lx = i - ly * W;
        edge[q] = i < N ? min(min(lx, W - 1 - lx), min(ly, H - 1 - ly)) : -1;
        if (i >= N) continue;
        int x = x0 + lx, y = y0 + ly;
        if (near) {
            x += x < 0 ? nx : (x >= nx ? -nx : 0);
            y += y < 0 ? ny : (y >= ny ? -ny : 0);
        } else {
            x = wrapd(x, nx);
            y = wrapd(y, ny);
        }
        const float* p = src + (long long)y * nx + x;
#pragma unroll
        for (int c = 0; c < 3; ++c) v[q][c] = __ldcg(p + c * NP);   // written by the previous pass
    }
#pragma unroll
    for (int q = 0; q < C; ++q)
        if (edge[q] >= 0)
#pragma unroll
            for (int c = 0; c < 3; ++c) sA[c * N + threadIdx.x + q * DNT] = v[q][c];
    __syncthreads();
#pragma unroll
    for (int s = 0; s < S; ++s) {
#pragma unroll
        for (int q = 0; q < C; ++q) {
            if (edge[q] < 2 * s + 1) continue;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float* a = sA + c * N + threadIdx.x + q * DNT;
                l0[q][c] = a[1] + a[-1] + a[W] + a[-W] - 4.f * v[q][c];
                sB[c * N + threadIdx.x + q * DNT] = v[q][c] + D * l0[q][c];
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < C; ++q) {
            if (edge[q] < 2 * s + 2) continue;
            const int i = threadIdx.x + q * DNT;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float* b = sB + c * N + i;
                const float l1 = b[1] + b[-1] + b[W] + b[-W] - 4.f * b[0];
                v[q][c] = v[q][c] + 0.5f * D * (l0[q][c] + l1);
                if (s < S - 1) sA[c * N + i] = v[q][c];
            }
            if (s == S - 1) {
                const int ly = i / W, lx = i - ly * W;
                const int gx = x0 + lx, gy = y0 + ly;
                if (gx >= nx || gy >= ny) continue;
                float* o = dst + (long long)gy * nx + gx;
#pragma unroll
                for (int c = 0; c < 3; ++c) o[c * NP] = v[q][c];
            }
        }
        __syncthreads();
    }
}

// pass k of d sub-steps on one tile, from the buffer whose turn it is to the other one
// (sig_new: the step's result, and the last pass's; sig_tmp: the other buffer); with d = 1 the
// second pass copies
__device__ __forceinline__ void diffuse_pass(float* sig_new, float* sig_tmp, long long NP, int nx, int ny, float D, int d,
                                             int k, int bx, int by, float* sm)
{
    const float* src = (k & 1) ? sig_tmp : sig_new;
    float* dst = (k & 1) ? sig_new : sig_tmp;
    switch (pass_steps(d, k)) {
    case 3: diffuse_steps<3>(src, dst, NP, nx, ny, D, bx, by, sm); break;
    case 2: diffuse_steps<2>(src, dst, NP, nx, ny, D, bx, by, sm); break;
    case 1: diffuse_steps<1>(src, dst, NP, nx, ny, D, bx, by, sm); break;
    default:
        for (int i = threadIdx.x; i < DX * DY; i += DNT) {
            const int gx = bx * DX + i % DX, gy = by * DY + i / DX;
            if (gx >= nx || gy >= ny) continue;
            const long long g = (long long)gy * nx + gx;
            for (int c = 0; c < 3; ++c) dst[c * NP + g] = __ldcg(src + c * NP + g);
        }
        __syncthreads();
    }
}

}  // namespace dif
}  // namespace vlb
