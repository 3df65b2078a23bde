// lb_batch.cu -- batched sweeps: many independent lattices of uneven sizes advanced together,
// a chunk of steps per captured CUDA graph.
//
// Default (phase launches): each step is one launch per phase and group of instances -- all
// instances' lattice tiles (k_batch_tiles, the tile kernel's occupancy of three CTAs per SM),
// then their diffusion passes beside their rings' node steps -- in stream order, so no kernel waits
// on another inside a launch.  A group holds instances of one tile shape, those with diffusion
// sub-steps apart from those without, which make two groups: instances are independent, so where there
// are several groups each has a stream of its own and its short launches run beside the lattice launches
// of the others (20 lattices of 128^2 to 512^2, 30 steps: 6109 -> 5500 us).
// Alternatively (lb_batch_set_persistent) one persistent cooperative kernel per group runs the whole
// chunk, each step having three phases separated by a grid barrier:
//   lattice  the fused step of every tile of every instance (tile shape per instance, chosen by
//            the autotuner among 32x16, 32x8, 64x8, 16x16), the tile code of lb_tile.cuh;
//   sigma    diffusion passes of the instances whose D_p exceeds the Heun bound;
//   nodes    the node step of every ring of every instance (lb_node.cuh).
// Work items are assigned to CTAs round-robin, so the schedule and every result are the same
// from run to run.  The barrier spins with an iteration limit and reports LB_ETIMEOUT.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "lb_diffuse.cuh"
#include "lb_handle.h"
#include "lb_node.cuh"
#include "lb_strip.cuh"
#include "lb_tile.cuh"

namespace vlb {
namespace {

constexpr int BT = 256;     // threads per CTA
static_assert(BT == dif::DNT, "a diffusion tile is a CTA of a batch kernel");
// tile shapes 0..3 (32x16, 32x8, 64x8, 16x16 cells per CTA), and shape 4: the warp-strip kernel
// (phase launches only; a CTA = SWARPS strips of SOWN columns x STRIP_H rows)
constexpr int N_SHAPES = 5;
constexpr int N_TILE_SHAPES = 4;
constexpr int SHAPE_STRIP = 4;
constexpr int STRIP_H = 64;
// groups: per shape two of instances without diffusion sub-steps, of about as many tiles (the node steps
// of the one run beside the tiles of the other), and one of those with (persistent launches: all in
// the first of the three)
constexpr int LANES = 3, LANE_SUB = 2;
constexpr int N_GROUPS = LANES * N_SHAPES;
static_assert(N_GROUPS < 32, "k_batch_parity takes a mask of groups");
constexpr int group_shape(int g) { return g / LANES; }
__host__ __device__ constexpr int shape_tx(int s) { return s == 0 ? 32 : (s == 1 ? 32 : (s == 2 ? 64 : 16)); }
__host__ __device__ constexpr int shape_ty(int s) { return s == 0 ? 16 : (s == 1 ? 8 : (s == 2 ? 8 : 16)); }

constexpr size_t cmaxz(size_t a, size_t b) { return a > b ? a : b; }
// dynamic shared memory of the kernel of one tile shape
template <int TX, int TY>
constexpr size_t batch_smem()
{
    return cmaxz(cmaxz(tile::TileGeo<TX, TY>::SMEM_BYTES, sizeof(float) * dif::SMEM), sizeof(node::NodeSmem));
}

struct BatchInst {
    FusedArgs fa[2];            // lattice step from buffer p to buffer p^1, p = 0, 1
    NodeArgs na;
    float* sig[2];              // sigma planes of buffer 0 and 1
    double2* xb[2];             // node positions read in a step whose lattice source is buffer p
    int shape, tiles_x, tiles_y;
    int dsub;                   // diffusion sub-steps (0: none)
    float dsub_D;               // D_p / dsub
    int dif_tx, dif_ty;
};

struct BatchArgs {
    const BatchInst* inst;
    int n_inst;
    const int* tile_begin;      // prefix sums of lattice tiles over instances (n_inst + 1)
    const int* tile_inst;       // instance of each lattice tile (phase launches)
    const int* node_begin;      // prefix sums of rings (one for an instance without)
    const int* dif_begin;       // prefix sums of diffusion tiles (instances with dsub > 0)
    int max_dsub;
    int* cur;                   // buffer parity of the current state (device)
    unsigned* bar;              // [0] arrivals, [1] generation
    int* err;                   // barrier timeout flag
    unsigned extra_arrivals;    // 0; > 0 only to exercise the timeout path
    unsigned long long wait_ns; // limit of one barrier wait
};

__device__ __forceinline__ int find_inst(const int* begin, int n, int item)
{
    int lo = 0, hi = n;          // begin[lo] <= item < begin[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (begin[mid] <= item) lo = mid; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier of a cooperative launch (all CTAs are co-resident).  The wait gives up after
// B.wait_ns (or 2^26 polls), sets the error flag and returns false; the caller then stops.
__device__ bool grid_sync(const BatchArgs& B)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned* gen = B.bar + 1;
        const unsigned g = *gen;
        __threadfence();
        int ok = 1;
        if (atomicAdd(B.bar, 1u) == gridDim.x - 1 + B.extra_arrivals) {
            B.bar[0] = 0u;
            __threadfence();
            atomicAdd(B.bar + 1, 1u);
        } else {
            const unsigned long long t0 = global_ns();
            unsigned it = 0;
            while (*gen == g) {
                if (++it > (1u << 26) || global_ns() - t0 > B.wait_ns) {
                    atomicExch(B.err, 1);
                    ok = 0;
                    break;
                }
                __nanosleep(100);
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// One kernel per tile shape: the instances of a batch are grouped by their shape and each group
// runs its own persistent launch (one tile body per kernel keeps within the register budget of
// two 256-thread CTAs per SM; the instances are independent, so the groups need no common
// barrier).
template <int TX, int TY, bool SCALAR>
__global__ void __launch_bounds__(BT, 2) k_batch(const BatchArgs B, int nsteps)
{
    extern __shared__ __align__(16) float sm[];
    const int cur0 = *B.cur;
    const int n_tiles = __ldg(B.tile_begin + B.n_inst), n_nodes = __ldg(B.node_begin + B.n_inst);
    const int n_dif = __ldg(B.dif_begin + B.n_inst);
    bool ok = true;
    for (int s = 0; s < nsteps && ok; ++s) {
        const int par = (cur0 + s) & 1;
        for (int item = blockIdx.x; item < n_tiles; item += gridDim.x) {
            const int i = find_inst(B.tile_begin, B.n_inst, item);
            const BatchInst& I = B.inst[i];
            const int local = item - __ldg(B.tile_begin + i);
            const int by = local / I.tiles_x, bx = local - by * I.tiles_x;
            // the tile step of lb_step; coherent loads: the state was written by the previous step
            // of this launch
            tile::tile_step<MODE_STEP, cell::PREC_FP32, TX, TY, true, SCALAR>(I.fa[par], bx, by, local, sm);
            __syncthreads();     // shared memory is reused by the next item
        }
        ok = grid_sync(B);
        // diffusion passes: sigma of the new buffer (par^1) and the old one as the other buffer
        for (int k = 0; k < dif::passes(B.max_dsub) && ok && n_dif > 0; ++k) {
            for (int item = blockIdx.x; item < n_dif; item += gridDim.x) {
                const int i = find_inst(B.dif_begin, B.n_inst, item);
                const BatchInst& I = B.inst[i];
                const int local = item - __ldg(B.dif_begin + i);
                const int by = local / I.dif_tx, bx = local - by * I.dif_tx;
                if (k < dif::passes(I.dsub))
                    dif::diffuse_pass(I.sig[par ^ 1], I.sig[par], I.fa[0].plane, I.fa[0].nx, I.fa[0].ny, I.dsub_D, I.dsub,
                                      k, bx, by, sm);
            }
            ok = grid_sync(B);
        }
        if (!ok) break;
        for (int item = blockIdx.x; item < n_nodes; item += gridDim.x) {
            const int i = find_inst(B.node_begin, B.n_inst, item);
            NodeArgs na = B.inst[i].na;
            na.X = B.inst[i].xb[par];
            na.X_out = B.inst[i].xb[par ^ 1];
            // the tiles' shared memory is free in this phase
            node::node_step(na, na.n_rings > 0 ? item - __ldg(B.node_begin + i) : -1, *reinterpret_cast<node::NodeSmem*>(sm));
            __syncthreads();
        }
        ok = grid_sync(B);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *B.cur = (cur0 + nsteps) & 1;
}

// ---- phase launches: one CTA per work item, the buffer parity of step s of the chunk read from
// the device word (so that a replayed graph continues from wherever the last chunk ended) ----

template <int TX, int TY, bool SCALAR>
__global__ void __launch_bounds__(BT, 3) k_batch_tiles(const BatchArgs B, int s)
{
    extern __shared__ __align__(16) float sm[];
    const int par = (*B.cur + s) & 1;
    const int item = blockIdx.x;
    // one load where a search among the prefix sums is log2 n dependent ones at the start of every CTA
    // (a sweep of 20 lattices, 30 steps: 5482 -> 5344 us)
    const int i = __ldg(B.tile_inst + item);
    const BatchInst& I = B.inst[i];
    const int local = item - __ldg(B.tile_begin + i);
    const int by = local / I.tiles_x, bx = local - by * I.tiles_x;
    // the state was written by an earlier launch: the read-only path is safe
    tile::tile_step<MODE_STEP, cell::PREC_FP32, TX, TY, false, SCALAR>(I.fa[par], bx, by, local, sm);
}

// the warp-strip step of every instance of the strip group: CTA `local` of an instance covers
// strip columns (local % tiles_x) * SWARPS .. and rows chunk local / tiles_x; the step index comes
// from the instance's control block (advanced by its node step of the step before)
template <bool SCALAR>
__global__ void __launch_bounds__(SNT, 3) k_batch_strips(const BatchArgs B, int s)
{
    extern __shared__ __align__(16) float smem[];
    const int par = (*B.cur + s) & 1;
    const int item = blockIdx.x;
    const int i = __ldg(B.tile_inst + item);
    const BatchInst& I = B.inst[i];
    const int local = item - __ldg(B.tile_begin + i);
    const int cy = local / I.tiles_x, cx = local - cy * I.tiles_x;
    strip_body<cell::PREC_FP32, SCALAR>(I.fa[par], I.fa[par].ctl->t, STRIP_H, cx, cy, local, smem);
}

// pass k of the diffusion of the instances with sub-steps (those of more passes than k)
__global__ void __launch_bounds__(BT) k_batch_diffuse(const BatchArgs B, int s, int k)
{
    extern __shared__ __align__(16) float sm[];
    const int par = (*B.cur + s) & 1;
    const int item = blockIdx.x;
    const int i = find_inst(B.dif_begin, B.n_inst, item);
    const BatchInst& I = B.inst[i];
    if (k >= dif::passes(I.dsub)) return;
    const int local = item - __ldg(B.dif_begin + i);
    const int by = local / I.dif_tx, bx = local - by * I.dif_tx;
    dif::diffuse_pass(I.sig[par ^ 1], I.sig[par], I.fa[0].plane, I.fa[0].nx, I.fa[0].ny, I.dsub_D, I.dsub, k, bx, by, sm);
}

__global__ void __launch_bounds__(NODE_THREADS) k_batch_nodes(const BatchArgs B, int s)
{
    __shared__ node::NodeSmem S;
    const int par = (*B.cur + s) & 1;
    const int item = blockIdx.x;
    const int i = find_inst(B.node_begin, B.n_inst, item);
    NodeArgs na = B.inst[i].na;
    na.X = B.inst[i].xb[par];
    na.X_out = B.inst[i].xb[par ^ 1];
    node::node_step(na, na.n_rings > 0 ? item - __ldg(B.node_begin + i) : -1, S);
}

// the buffer parities after a chunk of n steps: those of the groups in `mask` (every instance has
// the same one, so that a word is right for whichever group an instance comes to)
__global__ void k_batch_parity(int* cur, unsigned mask, int n)
{
    if (threadIdx.x < N_GROUPS && ((mask >> threadIdx.x) & 1u)) cur[threadIdx.x] = (cur[threadIdx.x] + n) & 1;
}

}  // namespace
}  // namespace vlb

using namespace vlb;

struct lb_batch {
    std::vector<lb_handle*> h;
    cudaStream_t user = nullptr;            // the handles' stream
    cudaStream_t stream = nullptr;          // the batch's own stream (capturable)
    cudaEvent_t ev_in = nullptr, ev_out = nullptr;
    std::vector<int> shape;                 // per instance
    bool scalar = false;                    // every instance runs the scalar model (else none does)
    // per group: device descriptors, prefix sums and work items, in one buffer sized for any shapes
    // (plan_cap), and (phase launches) its streams: the lattice and diffusion launches on one, the
    // node steps on the other
    char* d_plan = nullptr;
    size_t plan_cap = 0;
    bool planned = false;                   // the plan is complete (else no step runs)
    cudaStream_t main[N_GROUPS] = {}, side[N_GROUPS] = {};
    cudaEvent_t ev_main[N_GROUPS] = {}, ev_side[N_GROUPS] = {};
    BatchInst* d_inst[N_GROUPS] = {};
    int* d_tile_begin[N_GROUPS] = {};
    int* d_tile_inst[N_GROUPS] = {};
    int* d_node_begin[N_GROUPS] = {};
    int* d_dif_begin[N_GROUPS] = {};
    int n_group[N_GROUPS] = {};
    int max_dsub[N_GROUPS] = {};
    int n_tiles[N_GROUPS] = {};             // work items (phase launches)
    int n_nodes[N_GROUPS] = {};
    int n_dif[N_GROUPS] = {};
    int grid[N_SHAPES] = {};                // CTAs of each shape's persistent launch
    bool persistent = false;                // one persistent kernel per chunk (else phase launches)
    int* d_cur = nullptr;                   // buffer parity, one word per group
    unsigned* d_bar = nullptr;              // barrier words, two per group
    int* d_err = nullptr;
    std::vector<double*> partials;          // per instance: readout partial sums sized for any shape
    int chunk = 10;
    unsigned extra_arrivals = 0;
    unsigned long long wait_ns = 2000000000ull;
    cudaGraphExec_t graph = nullptr;
    bool graph_tried = false;
    std::string err;
};

namespace {

// the strip shape applies to this instance (the warp-strip kernel's conditions)
bool strip_ok(const lb_handle* h) { return strip_eligible(h->p.nx, h->p.ny, h->p.walls_x || h->p.walls_y); }

int bfail(lb_batch* b, int code, const std::string& msg)
{
    if (b) b->err = msg;
    return code;
}

#define BCK(b, call)                                                                   \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess) {                                                       \
            if (b) b->err = std::string(#call) + ": " + cudaGetErrorString(e_);        \
            return e_ == cudaErrorMemoryAllocation ? LB_ENOMEM : LB_ECUDA;             \
        }                                                                              \
    } while (0)

void drop_graph(lb_batch* b)
{
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
    b->graph_tried = false;
}

// work items of a lattice step of one instance, in x and y
void lattice_items(const lb_handle* h, int sh, int& tx, int& ty)
{
    if (sh == SHAPE_STRIP) {
        tx = ((h->p.nx + SOWN - 1) / SOWN + SWARPS - 1) / SWARPS;
        ty = (h->p.ny + STRIP_H - 1) / STRIP_H;
    } else {
        tx = (h->p.nx + shape_tx(sh) - 1) / shape_tx(sh);
        ty = (h->p.ny + shape_ty(sh) - 1) / shape_ty(sh);
    }
}

// bytes of the plan of these instances, whatever their shapes: descriptors, three prefix sums per group,
// the instance of every tile
size_t plan_bytes(const std::vector<lb_handle*>& hs)
{
    size_t ints = 3 * (hs.size() + N_GROUPS);
    for (const lb_handle* h : hs) {
        int most = 0;
        for (int sh = 0; sh < N_SHAPES; ++sh) {
            int tx, ty;
            lattice_items(h, sh, tx, ty);
            most = std::max(most, tx * ty);
        }
        ints += most;
    }
    return sizeof(BatchInst) * hs.size() + sizeof(int) * ints;
}

int groups_used(const lb_batch* b)
{
    int used = 0;
    for (int g = 0; g < N_GROUPS; ++g) used += b->n_group[g] > 0;
    return used;
}

// the node steps of a group run on a stream of their own: beside the group's diffusion or other groups
bool nodes_fork(const lb_batch* b, int g, int used) { return (b->n_dif[g] > 0 || used > 1) && b->n_nodes[g] > 0; }

// (re)build the per-instance descriptors of every shape group for the current tile shapes; nothing of the
// batch is in flight.  The former plan and its graph are gone first: when a call fails half way no step
// runs until a plan is complete.
int build_plan(lb_batch* b)
{
    drop_graph(b);
    b->planned = false;
    const int n = (int)b->h.size();
    std::vector<int> lane(n, 0);
    if (!b->persistent) {
        long long cells[N_SHAPES][2] = {};
        for (int i = 0; i < n; ++i) {
            long long* c = cells[b->shape[i]];
            if (b->h[i]->p.diffusion_substeps > 0) lane[i] = LANE_SUB;
            else {
                lane[i] = c[1] < c[0] ? 1 : 0;
                c[lane[i]] += b->h[i]->plane;
            }
        }
    }
    // the buffer: the descriptors of the groups one after the other, then each group's tables
    std::vector<char> plan(b->plan_cap);
    size_t inst_at = 0, int_at = sizeof(BatchInst) * (size_t)n;
    auto table = [&](const std::vector<int>& v) {
        memcpy(plan.data() + int_at, v.data(), sizeof(int) * v.size());
        int* d = reinterpret_cast<int*>(b->d_plan + int_at);
        int_at += sizeof(int) * v.size();
        return d;
    };
    for (int g = 0; g < N_GROUPS; ++g) {
        const int sh = group_shape(g);
        std::vector<BatchInst> inst;
        std::vector<int> tb(1, 0), nb(1, 0), db(1, 0), ti;
        b->max_dsub[g] = 0;
        for (int i = 0; i < n; ++i) {
            lb_handle* h = b->h[i];
            if (b->shape[i] != sh || lane[i] != g % LANES) continue;
            BatchInst I;
            const int save = h->cur;
            for (int p = 0; p < 2; ++p) {
                h->cur = p;
                I.fa[p] = handle_fused_args(h);
                I.fa[p].partials = b->partials[i];
            }
            h->cur = save;
            I.na = handle_node_args(h, 1);
            I.na.partials = b->partials[i];
            I.xb[h->cur] = h->X;
            I.xb[h->cur ^ 1] = h->X_alt;
            I.shape = sh;
            lattice_items(h, sh, I.tiles_x, I.tiles_y);
            I.na.n_partials = I.tiles_x * I.tiles_y;
            for (int p = 0; p < 2; ++p) I.sig[p] = static_cast<float*>(h->state[p]) + (size_t)PL_SXX * h->plane;
            I.dsub = h->p.diffusion_substeps;
            I.dsub_D = I.dsub > 0 ? (float)(h->p.Dp / I.dsub) : 0.f;
            I.dif_tx = diffuse_tiles_x(h->p.nx);
            I.dif_ty = diffuse_tiles_y(h->p.ny);
            b->max_dsub[g] = std::max(b->max_dsub[g], I.dsub);
            tb.push_back(tb.back() + I.tiles_x * I.tiles_y);
            ti.resize(tb.back(), (int)inst.size());
            nb.push_back(nb.back() + I.na.n_ctas);
            db.push_back(db.back() + (I.dsub > 0 ? I.dif_tx * I.dif_ty : 0));
            inst.push_back(I);
        }
        b->n_group[g] = (int)inst.size();
        b->n_tiles[g] = tb.back();
        b->n_nodes[g] = nb.back();
        b->n_dif[g] = db.back();
        if (inst.empty()) continue;
        b->d_inst[g] = reinterpret_cast<BatchInst*>(b->d_plan + inst_at);
        memcpy(plan.data() + inst_at, inst.data(), sizeof(BatchInst) * inst.size());
        inst_at += sizeof(BatchInst) * inst.size();
        b->d_tile_begin[g] = table(tb);
        b->d_node_begin[g] = table(nb);
        b->d_dif_begin[g] = table(db);
        b->d_tile_inst[g] = table(ti);
    }
    // the streams and events that launch_phases will use and that are not there yet
    const int used = groups_used(b);
    for (int g = 0; g < N_GROUPS && !b->persistent; ++g) {
        if (!b->n_group[g]) continue;
        // sub-stepped instances have the longest chain of launches, node steps are short and hold up
        // the next tiles: theirs go first
        int least = 0, greatest = 0;
        if (used > 1) {
            BCK(b, cudaDeviceGetStreamPriorityRange(&least, &greatest));
            if (!b->main[g])
                BCK(b, cudaStreamCreateWithPriority(&b->main[g], cudaStreamNonBlocking, g % LANES == LANE_SUB ? greatest : least));
            if (!b->ev_main[g]) BCK(b, cudaEventCreateWithFlags(&b->ev_main[g], cudaEventDisableTiming));
        }
        if (nodes_fork(b, g, used)) {
            BCK(b, cudaDeviceGetStreamPriorityRange(&least, &greatest));
            if (!b->side[g]) BCK(b, cudaStreamCreateWithPriority(&b->side[g], cudaStreamNonBlocking, greatest));
            if (!b->ev_side[g]) BCK(b, cudaEventCreateWithFlags(&b->ev_side[g], cudaEventDisableTiming));
        }
    }
    BCK(b, cudaMemcpy(b->d_plan, plan.data(), int_at, cudaMemcpyHostToDevice));
    b->planned = true;
    return LB_OK;
}

BatchArgs batch_args(const lb_batch* b, int g)
{
    BatchArgs a;
    a.inst = b->d_inst[g];
    a.n_inst = b->n_group[g];
    a.tile_begin = b->d_tile_begin[g];
    a.tile_inst = b->d_tile_inst[g];
    a.node_begin = b->d_node_begin[g];
    a.dif_begin = b->d_dif_begin[g];
    a.max_dsub = b->max_dsub[g];
    a.cur = b->d_cur + g;
    a.bar = b->d_bar + 2 * group_shape(g);
    a.err = b->d_err;
    a.extra_arrivals = b->extra_arrivals;
    a.wait_ns = b->wait_ns;
    return a;
}

template <int TX, int TY>
cudaError_t launch_shape(const lb_batch* b, int sh, int nsteps)
{
    BatchArgs a = batch_args(b, LANES * sh);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b->grid[sh]);
    cfg.blockDim = dim3(BT);
    cfg.dynamicSmemBytes = batch_smem<TX, TY>();
    cfg.stream = b->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return b->scalar ? cudaLaunchKernelEx(&cfg, k_batch<TX, TY, true>, a, nsteps)
                     : cudaLaunchKernelEx(&cfg, k_batch<TX, TY, false>, a, nsteps);
}

template <int TX, int TY>
cudaError_t launch_tiles(const lb_batch* b, int g, int s, cudaStream_t st)
{
    static unsigned long long attr_done = 0;     // per device
    auto kern = b->scalar ? k_batch_tiles<TX, TY, true> : k_batch_tiles<TX, TY, false>;
    const size_t smem = tile::TileGeo<TX, TY>::SMEM_BYTES;
    if (!done_on_device(attr_done)) {
        cudaError_t e = cudaFuncSetAttribute(k_batch_tiles<TX, TY, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_batch_tiles<TX, TY, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) {
            attr_done = 0;
            return e;
        }
    }
    kern<<<b->n_tiles[g], BT, smem, st>>>(batch_args(b, g), s);
    return cudaGetLastError();
}

cudaError_t launch_strips(const lb_batch* b, int g, int s, cudaStream_t st)
{
    static unsigned long long attr_done = 0;     // per device
    if (!done_on_device(attr_done)) {
        cudaError_t e = cudaFuncSetAttribute(k_batch_strips<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)STRIP_SMEM);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_batch_strips<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)STRIP_SMEM);
        if (e != cudaSuccess) {
            attr_done = 0;
            return e;
        }
    }
    auto kern = b->scalar ? k_batch_strips<true> : k_batch_strips<false>;
    kern<<<b->n_tiles[g], SNT, STRIP_SMEM, st>>>(batch_args(b, g), s);
    return cudaGetLastError();
}

// the lattice step of one group
cudaError_t launch_lattice(const lb_batch* b, int g, int s, cudaStream_t st)
{
    switch (group_shape(g)) {
    case 0: return launch_tiles<32, 16>(b, g, s, st);
    case 1: return launch_tiles<32, 8>(b, g, s, st);
    case 2: return launch_tiles<64, 8>(b, g, s, st);
    case 3: return launch_tiles<16, 16>(b, g, s, st);
    default: return launch_strips(b, g, s, st);
    }
}

// Phase launches of `nsteps` steps: per step and group the lattice step, then the diffusion passes
// beside the node steps (neither reads what the other writes); at the end the groups' streams
// join and the device parity words advance.  One group alone stays on the batch's stream.
cudaError_t launch_phases(const lb_batch* b, int nsteps)
{
    cudaError_t e = cudaSuccess;
    const size_t dsm = sizeof(float) * dif::SMEM;
    auto ok = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
        return e == cudaSuccess;
    };
    auto after = [&](cudaStream_t st, cudaEvent_t ev, cudaStream_t src) {     // st goes on when src is here
        return ok(cudaEventRecord(ev, src)) && ok(cudaStreamWaitEvent(st, ev, 0));
    };
    const int used = groups_used(b);
    cudaStream_t st[N_GROUPS];
    for (int g = 0; g < N_GROUPS; ++g) {
        st[g] = used > 1 ? b->main[g] : b->stream;
        if (b->n_group[g] && used > 1 && !after(st[g], b->ev_main[g], b->stream)) return e;
    }
    for (int s = 0; s < nsteps; ++s)
        for (int g = N_GROUPS - 1; g >= 0; --g) {
            if (!b->n_group[g]) continue;
            if (!ok(launch_lattice(b, g, s, st[g]))) return e;
            const bool fork = nodes_fork(b, g, used);
            if (b->n_nodes[g]) {
                if (fork && !after(b->side[g], b->ev_side[g], st[g])) return e;
                k_batch_nodes<<<b->n_nodes[g], NODE_THREADS, 0, fork ? b->side[g] : st[g]>>>(batch_args(b, g), s);
                if (!ok(cudaGetLastError())) return e;
            }
            for (int k = 0; b->n_dif[g] && k < dif::passes(b->max_dsub[g]); ++k) {
                k_batch_diffuse<<<b->n_dif[g], BT, dsm, st[g]>>>(batch_args(b, g), s, k);
                if (!ok(cudaGetLastError())) return e;
            }
            if (fork && !after(st[g], b->ev_side[g], b->side[g])) return e;
        }
    for (int g = 0; g < N_GROUPS; ++g)
        if (b->n_group[g] && used > 1 && !after(b->stream, b->ev_main[g], st[g])) return e;
    k_batch_parity<<<1, 32, 0, b->stream>>>(b->d_cur, (1u << N_GROUPS) - 1u, nsteps);
    ok(cudaGetLastError());
    return e;
}

// one persistent launch per non-empty shape group, one after another on the batch stream (or
// the phase launches)
cudaError_t launch_batch(const lb_batch* b, int nsteps)
{
    if (!b->persistent) return launch_phases(b, nsteps);
    cudaError_t e = cudaSuccess;
    if (b->n_group[0] && e == cudaSuccess) e = launch_shape<32, 16>(b, 0, nsteps);
    if (b->n_group[LANES] && e == cudaSuccess) e = launch_shape<32, 8>(b, 1, nsteps);
    if (b->n_group[2 * LANES] && e == cudaSuccess) e = launch_shape<64, 8>(b, 2, nsteps);
    if (b->n_group[3 * LANES] && e == cudaSuccess) e = launch_shape<16, 16>(b, 3, nsteps);
    unsigned others = 0;             // a persistent launch advances its own word
    for (int g = 0; g < N_GROUPS; ++g)
        if (!b->n_group[g]) others |= 1u << g;
    if (e == cudaSuccess) {
        k_batch_parity<<<1, 32, 0, b->stream>>>(b->d_cur, others, nsteps);
        e = cudaGetLastError();
    }
    return e;
}

// shared-memory opt-in and the co-resident grid of one shape's kernel
template <int TX, int TY>
cudaError_t setup_shape(lb_batch* b, int sh, int n_sm)
{
    const size_t smem = batch_smem<TX, TY>();
    auto kern = b->scalar ? k_batch<TX, TY, true> : k_batch<TX, TY, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, BT, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    b->grid[sh] = n_sm * per_sm;
    return cudaSuccess;
}

// Capture one persistent launch of `chunk` steps as a graph (once per plan).  If capture or
// instantiation is refused, the batch keeps launching the kernel directly.
void capture(lb_batch* b)
{
    b->graph_tried = true;
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    const cudaError_t e = launch_batch(b, b->chunk);
    const cudaError_t e2 = cudaStreamEndCapture(b->stream, &g);
    if (e == cudaSuccess && e2 == cudaSuccess && g && cudaGraphInstantiate(&b->graph, g, cudaGraphInstantiateFlagUseNodePriority) != cudaSuccess)
        b->graph = nullptr;
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();
}

// n steps on the batch stream, ordered after the work already queued on the handles' stream and
// before anything queued there later
int run_steps(lb_batch* b, long long n)
{
    if (n == 0) return LB_OK;
    if (!b->planned) return bfail(b, LB_ESTATE, "no complete plan: set the shapes again");
    if (!b->graph_tried) capture(b);
    BCK(b, cudaEventRecord(b->ev_in, b->user));
    BCK(b, cudaStreamWaitEvent(b->stream, b->ev_in, 0));
    long long left = n;
    while (b->graph && left >= b->chunk) {
        BCK(b, cudaGraphLaunch(b->graph, b->stream));
        left -= b->chunk;
    }
    while (left > 0) {
        const int k = (int)std::min<long long>(left, b->chunk);
        BCK(b, launch_batch(b, k));
        left -= k;
    }
    BCK(b, cudaEventRecord(b->ev_out, b->stream));
    BCK(b, cudaStreamWaitEvent(b->user, b->ev_out, 0));
    for (lb_handle* h : b->h) {
        h->t += n;
        h->cur ^= (int)(n & 1);
        if (n & 1) std::swap(h->X, h->X_alt);
    }
    return LB_OK;
}

}  // namespace

extern "C" {

int lb_batch_create(lb_handle* const* handles, int32_t n, lb_batch** out)
{
    if (!handles || n < 1 || !out) return LB_EINVAL;
    *out = nullptr;
    for (int i = 0; i < n; ++i) {
        const lb_handle* h = handles[i];
        if (!h || !h->fields_ready || !h->body_ok) return LB_ESTATE;
        if (h->p.precision != LB_FP32 || h->p.model != handles[0]->p.model || h->cur != handles[0]->cur ||
            h->stream != handles[0]->stream)
            return LB_EINVAL;
        for (int k = 0; k < i; ++k)
            if (handles[k] == h) return LB_EINVAL;
    }
    lb_batch* b = new lb_batch();
    b->h.assign(handles, handles + n);
    for (lb_handle* h : b->h) ++h->batch_refs;   // its graphs hold the handles' state buffers
    b->user = handles[0]->stream;
    b->chunk = std::max(1, handles[0]->p.readout_every);
    b->shape.assign(n, 0);
    b->scalar = handles[0]->p.model == LB_MODEL_SCALAR;
    auto cleanup = [&](int code) { lb_batch_destroy(b); return code; };
    if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->ev_out, cudaEventDisableTiming) != cudaSuccess)
        return cleanup(LB_ECUDA);
    b->plan_cap = plan_bytes(b->h);
    if (cudaMalloc(&b->d_plan, b->plan_cap) != cudaSuccess) return cleanup(LB_ENOMEM);
    if (cudaMalloc(&b->d_cur, sizeof(int) * N_GROUPS) != cudaSuccess ||
        cudaMalloc(&b->d_bar, 2 * sizeof(unsigned) * N_SHAPES) != cudaSuccess ||
        cudaMalloc(&b->d_err, sizeof(int)) != cudaSuccess)
        return cleanup(LB_ENOMEM);
    for (int i = 0; i < n; ++i) {
        // enough partial sums for the smallest tile (16 x 8 cells covers every shape's count)
        double* p = nullptr;
        const long long tiles = ((long long)b->h[i]->p.nx / 16 + 1) * ((long long)b->h[i]->p.ny / 8 + 1);
        if (cudaMalloc(&p, sizeof(double) * 5 * tiles) != cudaSuccess) return cleanup(LB_ENOMEM);
        b->partials.push_back(p);
    }
    // the handles' queued work must be done before the batch's control words are set
    if (cudaStreamSynchronize(b->user) != cudaSuccess) return cleanup(LB_ECUDA);
    int cur[N_GROUPS];
    std::fill(cur, cur + N_GROUPS, handles[0]->cur);
    if (cudaMemcpy(b->d_cur, cur, sizeof cur, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(b->d_bar, 0, 2 * sizeof(unsigned) * N_SHAPES) != cudaSuccess ||
        cudaMemset(b->d_err, 0, sizeof(int)) != cudaSuccess)
        return cleanup(LB_ECUDA);
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (setup_shape<32, 16>(b, 0, n_sm) != cudaSuccess || setup_shape<32, 8>(b, 1, n_sm) != cudaSuccess ||
        setup_shape<64, 8>(b, 2, n_sm) != cudaSuccess || setup_shape<16, 16>(b, 3, n_sm) != cudaSuccess)
        return cleanup(LB_ECUDA);
    const int rc = build_plan(b);
    if (rc != LB_OK) return cleanup(rc);
    *out = b;
    return LB_OK;
}

int lb_batch_set_shape(lb_batch* b, int32_t inst, int32_t shape)
{
    if (!b) return LB_EINVAL;
    if (inst < -1 || inst >= (int)b->h.size() || shape < 0 || shape >= N_SHAPES)
        return bfail(b, LB_EINVAL, "bad instance or shape");
    if (shape == SHAPE_STRIP) {
        if (b->persistent) return bfail(b, LB_EINVAL, "the strip shape runs with phase launches only");
        for (int i = 0; i < (int)b->h.size(); ++i)
            if ((inst < 0 || i == inst) && !strip_ok(b->h[i]))
                return bfail(b, LB_EINVAL, "instance " + std::to_string(i) + " cannot take the strip shape "
                             "(periodic, nx >= 64 even, ny >= 32)");
    }
    BCK(b, cudaStreamSynchronize(b->stream));
    if (inst < 0) std::fill(b->shape.begin(), b->shape.end(), shape);
    else b->shape[inst] = shape;
    return build_plan(b);
}

int32_t lb_batch_shape(const lb_batch* b, int32_t inst)
{
    return b && inst >= 0 && inst < (int)b->h.size() ? b->shape[inst] : -1;
}

int lb_batch_step(lb_batch* b, int64_t n)
{
    if (!b) return LB_EINVAL;
    if (n < 0) return bfail(b, LB_EINVAL, "n < 0");
    return run_steps(b, n);
}

int lb_batch_sync(lb_batch* b)
{
    if (!b) return LB_EINVAL;
    BCK(b, cudaStreamSynchronize(b->stream));
    BCK(b, cudaStreamSynchronize(b->user));
    int e = 0;
    BCK(b, cudaMemcpy(&e, b->d_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (e) {
        const int z = 0;
        unsigned zb[2 * N_SHAPES] = {};
        BCK(b, cudaMemcpy(b->d_err, &z, sizeof(int), cudaMemcpyHostToDevice));
        BCK(b, cudaMemcpy(b->d_bar, zb, sizeof zb, cudaMemcpyHostToDevice));
        return bfail(b, LB_ETIMEOUT, "a grid barrier of the batched kernel timed out; the states are undefined");
    }
    for (size_t i = 0; i < b->h.size(); ++i) {
        const int rc = lb_sync(b->h[i]);
        if (rc != LB_OK) return bfail(b, rc, "instance " + std::to_string(i) + ": " + lb_last_error(b->h[i]));
    }
    return LB_OK;
}

int32_t lb_batch_grid(const lb_batch* b)
{
    if (!b) return 0;
    if (b->persistent) return b->grid[0];
    int n = 0;
    for (int g = 0; g < N_GROUPS; ++g) n += b->n_group[g] ? b->n_tiles[g] : 0;
    return n;
}

int lb_batch_set_persistent(lb_batch* b, int32_t enable)
{
    if (!b) return LB_EINVAL;
    if (enable != 0 && enable != 1) return bfail(b, LB_EINVAL, "enable must be 0 or 1");
    BCK(b, cudaStreamSynchronize(b->stream));
    if (enable)
        for (int sh : b->shape)
            if (sh == SHAPE_STRIP) return bfail(b, LB_EINVAL, "an instance has the strip shape (phase launches only)");
    b->persistent = enable != 0;
    return build_plan(b);
}

int32_t lb_batch_uses_graph(const lb_batch* b) { return b && b->graph ? 1 : 0; }

int lb_batch_set_wait_limit(lb_batch* b, double wait_ms, int32_t extra_arrivals)
{
    if (!b) return LB_EINVAL;
    if (!(wait_ms > 0.0 && wait_ms <= 60000.0) || extra_arrivals < 0)
        return bfail(b, LB_EINVAL, "need 0 < wait_ms <= 60000 and extra_arrivals >= 0");
    BCK(b, cudaStreamSynchronize(b->stream));
    b->wait_ns = (unsigned long long)(wait_ms * 1e6);
    b->extra_arrivals = (unsigned)extra_arrivals;
    drop_graph(b);
    return LB_OK;
}

// Autotuner: for every distinct lattice size of the batch, time `steps` batch steps with each
// tile shape applied to that size (the others unchanged) and keep the fastest.  The state is
// saved before and restored after, so tuning does not advance the simulation.  With a cache
// path, sizes already tuned on this GPU model are read from it and new results written back.
int lb_batch_autotune(lb_batch* b, const char* cache_path, int32_t steps)
{
    if (!b) return LB_EINVAL;
    if (steps < 1) return bfail(b, LB_EINVAL, "steps < 1");
    BCK(b, cudaStreamSynchronize(b->user));
    BCK(b, cudaStreamSynchronize(b->stream));
    cudaDeviceProp prop;
    int dev = 0;
    BCK(b, cudaGetDevice(&dev));
    BCK(b, cudaGetDeviceProperties(&prop, dev));
    std::map<std::string, int> cache;
    if (cache_path) {
        // flat JSON object, one entry per line:  "<gpu>|<nx>x<ny>": <shape>
        if (FILE* f = fopen(cache_path, "r")) {
            char line[512];
            while (fgets(line, sizeof line, f)) {
                char* q1 = strchr(line, '"');
                char* q2 = q1 ? strchr(q1 + 1, '"') : nullptr;
                int v = -1;
                if (q1 && q2 && sscanf(q2 + 1, " : %d", &v) == 1 && v >= 0 && v < N_SHAPES)
                    cache[std::string(q1 + 1, q2)] = v;
            }
            fclose(f);
        }
    }
    auto key_of = [&](const lb_handle* h) {
        return std::string(prop.name) + "|" + std::to_string(h->p.nx) + "x" + std::to_string(h->p.ny);
    };
    std::map<std::string, std::vector<int>> classes;
    for (int i = 0; i < (int)b->h.size(); ++i) classes[key_of(b->h[i])].push_back(i);
    bool need_tune = false;
    for (auto& kv : classes)
        if (!cache.count(kv.first)) need_tune = true;
    // snapshot everything a step writes: both state buffers, control words, series, nodes, rings
    std::vector<std::pair<void*, void*>> saved;      // (live, copy)
    std::vector<size_t> saved_bytes;
    auto release = [&]() {
        for (auto& s : saved) cudaFree(s.second);
        saved.clear();
    };
    if (need_tune) {
        for (lb_handle* h : b->h) {
            const size_t sb = (size_t)h->esz * N_PLANES * h->plane;
            std::vector<std::pair<void*, size_t>> items = {
                {h->state[0], sb}, {h->state[1], sb}, {h->ctl, sizeof(Ctl)},
                {h->series, sizeof(double) * (size_t)h->series_cap * h->row_len}};
            if (h->n_total > 0) {
                items.push_back({h->X, sizeof(double2) * h->n_total});
                items.push_back({h->node_cell, sizeof(int2) * h->n_total});
                items.push_back({h->node_frac, sizeof(float2) * h->n_total});
                items.push_back({h->node_force, sizeof(float2) * h->n_total});
                items.push_back({h->rings, sizeof(RingDev) * h->n_rings});
            }
            for (auto& it : items) {
                void* d = nullptr;
                if (cudaMalloc(&d, it.second) != cudaSuccess) {
                    release();
                    return bfail(b, LB_ENOMEM, "autotune snapshot");
                }
                saved.push_back({it.first, d});
                saved_bytes.push_back(it.second);
                if (cudaMemcpy(d, it.first, it.second, cudaMemcpyDeviceToDevice) != cudaSuccess) {
                    release();
                    return bfail(b, LB_ECUDA, "autotune snapshot copy");
                }
            }
        }
    }
    int dcur[N_GROUPS] = {};
    BCK(b, cudaMemcpy(dcur, b->d_cur, sizeof dcur, cudaMemcpyDeviceToHost));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    int rc = LB_OK;
    // time `steps` batch steps with the current shapes (after one warm-up step); < 0 on error
    auto time_plan = [&]() -> float {
        if ((rc = build_plan(b)) != LB_OK) return -1.f;
        cudaError_t e = launch_batch(b, 1);
        if (e == cudaSuccess) e = cudaEventRecord(e0, b->stream);
        if (e == cudaSuccess) e = launch_batch(b, steps);
        if (e == cudaSuccess) e = cudaEventRecord(e1, b->stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        float ms = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e != cudaSuccess) {
            rc = bfail(b, LB_ECUDA, std::string("autotune launch: ") + cudaGetErrorString(e));
            return -1.f;
        }
        return ms;
    };
    auto allowed = [&](int sh, int i) { return sh != SHAPE_STRIP || (!b->persistent && strip_ok(b->h[i])); };
    // First one shape for every untuned instance (one launch per phase for the whole batch: a
    // shape can pay only when most of the batch takes it), then each size class on its own from
    // there, the other classes fixed.
    if (need_tune) {
        float best = 3.0e38f;
        int best_s = 0;
        for (int sh = 0; sh < N_SHAPES && rc == LB_OK; ++sh) {
            bool ok = true;
            for (auto& kv : classes)
                if (!cache.count(kv.first))
                    for (int i : kv.second) ok = ok && allowed(sh, i);
            if (!ok) continue;
            for (auto& kv : classes) {
                auto hit = cache.find(kv.first);
                for (int i : kv.second) b->shape[i] = hit != cache.end() ? hit->second : sh;
            }
            const float ms = time_plan();
            if (ms >= 0.f && ms < best) {
                best = ms;
                best_s = sh;
            }
        }
        for (auto& kv : classes)
            if (!cache.count(kv.first))
                for (int i : kv.second) b->shape[i] = best_s;
    }
    for (auto& kv : classes) {
        if (rc != LB_OK) break;
        auto hit = cache.find(kv.first);
        if (hit != cache.end()) {
            for (int i : kv.second) b->shape[i] = hit->second;
            continue;
        }
        const int start = b->shape[kv.second[0]];
        float best = time_plan();
        int best_s = start;
        for (int sh = 0; sh < N_SHAPES && rc == LB_OK; ++sh) {
            if (sh == start || !allowed(sh, kv.second[0])) continue;
            for (int i : kv.second) b->shape[i] = sh;
            const float ms = time_plan();
            if (ms >= 0.f && ms < best) {
                best = ms;
                best_s = sh;
            }
        }
        for (int i : kv.second) b->shape[i] = best_s;
        cache[kv.first] = best_s;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    // restore the states, the device parity and the barrier words
    for (size_t k = 0; k < saved.size(); ++k)
        cudaMemcpy(saved[k].first, saved[k].second, saved_bytes[k], cudaMemcpyDeviceToDevice);
    release();
    cudaMemcpy(b->d_cur, dcur, sizeof dcur, cudaMemcpyHostToDevice);
    int berr = 0;
    cudaMemcpy(&berr, b->d_err, sizeof(int), cudaMemcpyDeviceToHost);
    if (rc != LB_OK) return rc;
    if (berr) return bfail(b, LB_ETIMEOUT, "a grid barrier timed out while tuning");
    rc = build_plan(b);
    if (rc != LB_OK) return rc;
    if (cache_path && need_tune) {
        if (FILE* f = fopen(cache_path, "w")) {
            fprintf(f, "{\n");
            size_t k = 0;
            for (auto& kv : cache)
                fprintf(f, "  \"%s\": %d%s\n", kv.first.c_str(), kv.second, ++k < cache.size() ? "," : "");
            fprintf(f, "}\n");
            fclose(f);
        } else {
            return bfail(b, LB_EINVAL, std::string("cannot write the tuning cache ") + cache_path);
        }
    }
    return LB_OK;
}

const char* lb_batch_last_error(const lb_batch* b) { return b ? b->err.c_str() : "null batch"; }

void lb_batch_destroy(lb_batch* b)
{
    if (!b) return;
    for (lb_handle* h : b->h) --h->batch_refs;
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->ev_in) cudaEventDestroy(b->ev_in);
    if (b->ev_out) cudaEventDestroy(b->ev_out);
    if (b->stream) cudaStreamDestroy(b->stream);
    for (int g = 0; g < N_GROUPS; ++g) {
        if (b->ev_main[g]) cudaEventDestroy(b->ev_main[g]);
        if (b->ev_side[g]) cudaEventDestroy(b->ev_side[g]);
        if (b->main[g]) cudaStreamDestroy(b->main[g]);
        if (b->side[g]) cudaStreamDestroy(b->side[g]);
    }
    cudaFree(b->d_plan);
    cudaFree(b->d_cur);
    cudaFree(b->d_bar);
    cudaFree(b->d_err);
    for (double* p : b->partials) cudaFree(p);
    delete b;
}

}  // extern "C"
