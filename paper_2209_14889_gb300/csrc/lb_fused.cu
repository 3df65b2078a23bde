// lb_fused.cu -- the tile kernels: one CTA per 32 x 16 tile of the fused step (lb_tile.cuh), one
// cell per thread (tile_step) or two neighbouring cells per thread on paired FP32 instructions
// (tile_step2); optionally with the node step of the same time step in their tail.
#include <cuda_runtime.h>

#include <cmath>

#include "lb_node.cuh"
#include "lb_tile.cuh"

namespace vlb {

namespace {

using namespace tile;

// One of n arrivals; true for the last, which leaves the counter at zero.  Release and acquire in
// the one atomic: a fence, an atomic, a store of the zero and a second fence took 3 200 cycles of
// the chain between the last tile and the ring's nodes.
__device__ __forceinline__ bool arrive(unsigned* counter, unsigned n)
{
    unsigned prev;
    asm volatile("atom.acq_rel.gpu.global.inc.u32 %0, [%1], %2;" : "=r"(prev) : "l"(counter), "r"(n - 1u) : "memory");
    return prev == n - 1u;
}

// The node step in the tail of the lattice kernel (FusedArgs::node_tail), after this tile's
// step (App. A).  A ring's nodes are read (spreading) only by the tiles whose region meets its
// box of step t, and the node update writes only the box of step t + 1 (RingDev::box), the
// nodes and the other position buffer: so once the last of those tiles has written u(t) and
// f^p(t) onto the box, the ring can advance while the remaining tiles run.  That tile advances
// it (node_ring), in the tile's shared memory, whose staged fields are dead by then.  On readout
// steps every tile counts itself and the last one sums the lattice readout.  A thread's arrival
// stands for the whole CTA: the barrier orders the CTA's writes before its fence.  Out of line:
// node_tail below calls it only for the tiles that have something to do.
template <int TX, int TY, bool EARLY>
__device__ __noinline__ void node_tail_work(const FusedArgs& a, float* sm, unsigned meet)
{
    using G = TileGeo<TX, TY>;
    node::NodeSmem& S = *reinterpret_cast<node::NodeSmem*>(sm);
    const int tid = threadIdx.x;
    const int nr = a.n_rings;
    const long long t = a.t;
    const int bx = blockIdx.x;
    int by = blockIdx.y + a.tile_rot;
    if (by >= (int)gridDim.y) by -= gridDim.y;
    if constexpr (EARLY) {
        const int* ar = reinterpret_cast<const int*>(sm + G::OFF_AR);
        __syncthreads();        // the tile's shared memory is free, AR_LAST is known
        if (ar[AR_COUNT] != 0) {
            meet = 0u;
            if (ar[AR_LAST]) {
                node::RingRegs rg;
                const int r = ar[AR_RING];
                rg.n = ar[AR_NODES];
                rg.off = ar[AR_OFF];
                rg.cap_w = ar[AR_CAP_W];
                rg.cap_h = ar[AR_CAP_H];
                rg.trap = ar[AR_TRAP] != 0;
                rg.box_off = *reinterpret_cast<const long long*>(ar + AR_BOX_OFF);
                rg.B = *reinterpret_cast<const int4*>(ar + AR_BOX);
                node::load_first_node(a.na, rg);
                __syncthreads();        // the node step's shared memory lies over these values
                node::node_ring(a.na, r, rg, S, t, (t % a.every) == 0);
            }
        }
    }
    for (int r = 0; r < nr && meet != 0u; ++r) {
        if (nr <= 32 && !((meet >> r) & 1u)) continue;
        const int4 B = ring_box(a.rings[r], t);
        if (nr > 32 &&
            (!meets(bx * TX - 2, G::R2W, B.x, B.z, a.nx) || !meets(by * TY - 2, G::R2H, B.y, B.w, a.ny)))
            continue;
        node::RingRegs rg;      // every tile that meets the ring loads what the last one needs
        node::load_ring(a.na, r, t, rg);
        node::load_first_node(a.na, rg);
        unsigned c = 0u;
        if (tid < 32)
            c = tiles_meeting(gridDim.x, TX, G::R2W, B.x, B.z, a.nx) *
                tiles_meeting(gridDim.y, TY, G::R2H, B.y, B.w, a.ny);
        __syncthreads();        // the tile's writes are out, its shared memory is free
        if (tid == 0) S.flag = arrive(&a.box_tickets[r], c);
        __syncthreads();
        if (S.flag) node::node_ring(a.na, r, rg, S, t, (t % a.every) == 0);
    }
    if ((t % a.every) == 0) {
        __syncthreads();
        if (tid == 0) S.flag = arrive(&a.ctl->tile_ticket, gridDim.x * gridDim.y);
        __syncthreads();
        if (S.flag) node::lattice_readout(a.na, t, S.dred);
    }
}

// The node tail of one tile: the step counter (one tile), then node_tail_work where this tile
// meets a ring's box or the step is a readout step; nothing else for most tiles.
template <int TX, int TY, bool EARLY = false>
__device__ __forceinline__ void node_tail(const FusedArgs& a, float* sm)
{
    using G = TileGeo<TX, TY>;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) a.ctl->t = a.t + 1;   // nothing here reads it
    // the rings whose box meets this tile's staged region (tested in ib_gather for up to 32 rings)
    const unsigned meet =
        a.n_rings > 32 ? 0xffffffffu : (unsigned)reinterpret_cast<const int*>(sm + G::OFF_SC)[NT / 32 + 2];
    if (meet != 0u || (a.t % a.every) == 0) node_tail_work<TX, TY, EARLY>(a, sm, meet);
}

// dynamic shared memory of a tile kernel: the tile's, or a ring's node step after it
template <int TX, int TY>
constexpr size_t tile_smem()
{
    return TileGeo<TX, TY>::SMEM_BYTES > sizeof(node::NodeSmem) ? TileGeo<TX, TY>::SMEM_BYTES : sizeof(node::NodeSmem);
}

template <int MODE, int PREC, bool SCALAR, int TX, int TY>
__global__ void __launch_bounds__(NT, 3) k_fused(const __grid_constant__ FusedArgs a)
{
    extern __shared__ __align__(16) float sm[];
    const bool tail = MODE == MODE_STEP && a.node_tail;
    int by = blockIdx.y;
    if (tail) {
        // consecutive lattice launches: the state staged first was written by the previous one
        pdl_wait();
        by += a.tile_rot;
        if (by >= (int)gridDim.y) by -= gridDim.y;
    }
    constexpr bool EARLY = MODE == MODE_STEP && TX * TY <= 128;
    tile_step<MODE, PREC, TX, TY, false, SCALAR, EARLY>(a, blockIdx.x, by, by * gridDim.x + blockIdx.x, sm);
    if (tail) node_tail<TX, TY, EARLY>(a, sm);
}

template <int MODE, int PREC>
__global__ void __launch_bounds__(NT, 2) k_fused_pair(const __grid_constant__ FusedArgs a)
{
    extern __shared__ __align__(16) float sm[];
    const bool tail = MODE == MODE_STEP && a.node_tail;
    int by = blockIdx.y;
    if (tail) {
        pdl_wait();
        by += a.tile_rot;
        if (by >= (int)gridDim.y) by -= gridDim.y;
    }
    tile_step2<MODE, PREC, TILE_X, TILE_Y>(a, blockIdx.x, by, by * gridDim.x + blockIdx.x, sm);
    if (tail) node_tail<TILE_X, TILE_Y>(a, sm);
}

// rho - rho0 needs the populations alone: streaming them takes the time of one pass over nine planes,
// the moments pass of the tile kernel (forces and all) six times as long.
template <int PREC>
__global__ void __launch_bounds__(256) k_drho(const void* src, float* out, long long NP, Phys ph)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= NP) return;
    float d[9];
#pragma unroll
    for (int n = 0; n < 9; ++n) d[n] = cell::ld_pop<PREC, false>(src, NP, n, g);
    float drho, ux, uy;
    cell::moments(ph, d, 0.f, 0.f, drho, ux, uy);
    out[g] = drho;
}

}  // namespace

cudaError_t launch_drho(const FusedArgs& a, float* out, cudaStream_t s)
{
    const unsigned n = (unsigned)((a.plane + 255) / 256);
    if (a.prec != PREC_FP32) k_drho<PREC_LP><<<n, 256, 0, s>>>(a.src, out, a.plane, a.ph);
    else k_drho<PREC_FP32><<<n, 256, 0, s>>>(a.src, out, a.plane, a.ph);
    return cudaGetLastError();
}

// Tile shapes of the one-cell step: 32x16, 16x16, 16x8, 8x8.
constexpr int SHAPE_X[FUSED_SHAPES] = {TILE_X, 16, 16, 8};
constexpr int SHAPE_Y[FUSED_SHAPES] = {TILE_Y, 16, 8, 8};

int fused_ctas(int nx, int ny, int shape)
{
    return ((nx + SHAPE_X[shape] - 1) / SHAPE_X[shape]) * ((ny + SHAPE_Y[shape] - 1) / SHAPE_Y[shape]);
}

// A lattice of few tiles is bound by the time of one tile (its passes of 256 threads over its regions,
// with a barrier and the loads' latency in each), so small tiles win until they fill the SMs several
// times over and the recomputed halo counts.  Measured on GB300 (us per step with one ring, shapes
// 0 .. 3): tensorial 32^2 without a ring 8.5, 6.5, 5.0, 4.7; 64^2 23.1, 19.8, 18.2, 17.3; 128^2 24.8,
// 20.9, 18.7, 19.0; 256^2 24.1, 22.2, 19.6, 19.8; 320^2 25.9, 23.5, 22.2, 24.9; 384^2 28.0, 27.3, 28.5,
// 39.6; 512^2 31.2, 31.5, 35.6, 52.8; 1024^2 61.3, 79.2, 107.9, 184.7.  The scalar model does half the
// work per cell: 384^2 29.4, 26.4, 24.3, 25.7; 512^2 29.2, 26.7, 26.0, 39.1; 640^2 30.7, 28.6, 34.4,
// 58.0; 768^2 31.5, 36.8, 47.3, 81.8.  Hence the limits, in tiles per SM: 8x8 up to 1, 16x8 up to 6
// (scalar 14), 16x16 up to 4 (scalar 12).
// Without a ring a tile is shorter by the gather and the node step, and the halo counts sooner: tensorial
// 96^2 9.0, 6.9, 5.3, 5.1; 224^2 9.1, 7.8, 7.0, 10.3; 250^2 9.1, 9.7, 10.4, 13.8; 320^2 10.8, 9.5, 12.1,
// 18.7; 384^2 13.5, 14.3, 16.3, 26.2; scalar 224^2 7.3, 6.3, 5.7, 8.7; 250^2 7.3, 7.8, 8.2, 11.8; 320^2 8.1,
// 7.5, 9.4, 15.6; 512^2 14.8, 16.9, 20.5, 34.3.  8x8 up to one tile per SM, 16x8 up to 3; beyond, 16x16 up
// to 3 where 32x16 tiles would take a second wave.
int fused_shape(int nx, int ny, int n_sm, bool scalar, bool rings)
{
    if (fused_ctas(nx, ny, 3) <= n_sm) return 3;
    if (!rings) {
        if (fused_ctas(nx, ny, 2) <= 3 * n_sm) return 2;
        return fused_ctas(nx, ny, 0) > n_sm && fused_ctas(nx, ny, 1) <= 3 * n_sm ? 1 : 0;
    }
    if (fused_ctas(nx, ny, 2) <= (scalar ? 14 : 6) * n_sm) return 2;
    if (fused_ctas(nx, ny, 1) <= (scalar ? 12 : 4) * n_sm) return 1;
    return 0;
}

int fused_tile_rot(int nx, int ny, double y_top)
{
    (void)nx;
    const int ty = (ny + TILE_Y - 1) / TILE_Y;
    int row = (int)std::floor(y_top / TILE_Y) % ty;
    if (row < 0) row += ty;
    return row;
}

template <int MODE, int PREC, bool PAIR, bool SCALAR = false, int TX = TILE_X, int TY = TILE_Y>
static cudaError_t launch_one(FusedArgs a, cudaStream_t s, bool pdl)
{
    static unsigned long long attr_done = 0;     // per device
    auto kern = [] {
        if constexpr (PAIR) return k_fused_pair<MODE, PREC>;
        else return k_fused<MODE, PREC, SCALAR, TX, TY>;
    }();
    if (!done_on_device(attr_done)) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tile_smem<TX, TY>());
        if (e != cudaSuccess) {
            attr_done = 0;
            return e;
        }
    }
    a.tile_rot = a.tile_rot * TILE_Y / TY;       // given in rows of TILE_Y cells
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.nx + TX - 1) / TX, (a.ny + TY - 1) / TY);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = tile_smem<TX, TY>();
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// the one-cell step with tiles of one shape
template <int PREC, bool SCALAR>
static cudaError_t launch_step(const FusedArgs& a, int shape, cudaStream_t s, bool pdl)
{
    switch (shape) {
    case 1: return launch_one<MODE_STEP, PREC, false, SCALAR, 16, 16>(a, s, pdl);
    case 2: return launch_one<MODE_STEP, PREC, false, SCALAR, 16, 8>(a, s, pdl);
    case 3: return launch_one<MODE_STEP, PREC, false, SCALAR, 8, 8>(a, s, pdl);
    default: return launch_one<MODE_STEP, PREC, false, SCALAR>(a, s, pdl);
    }
}

cudaError_t launch_fused(const FusedArgs& a, int mode, cudaStream_t s, int shape, bool pdl, bool pair)
{
    const bool lp = a.prec != PREC_FP32;
    if (mode == MODE_MOMENTS)
        return lp ? launch_one<MODE_MOMENTS, PREC_LP, false>(a, s, false) : launch_one<MODE_MOMENTS, PREC_FP32, false>(a, s, false);
    if (pair) return lp ? launch_one<MODE_STEP, PREC_LP, true>(a, s, pdl) : launch_one<MODE_STEP, PREC_FP32, true>(a, s, pdl);
    if (lp) return launch_step<PREC_LP, false>(a, shape, s, pdl);
    // the scalar model's step (FP32 state, one-cell tiles); its moments pass is the tensorial one,
    // which reads the unchanged P planes and, with the Ericksen force off, does not use them
    return a.scalar ? launch_step<PREC_FP32, true>(a, shape, s, pdl) : launch_step<PREC_FP32, false>(a, shape, s, pdl);
}

}  // namespace vlb
