// lb_node.cuh -- the node step (device code shared by the node kernel, the tail of the tile
// kernels and the batched kernels; App. A).
//
// Per step, after the lattice kernel of the same step has written u(t) (and, on readout steps,
// f^p(t)) onto the ring's work box:
//   * readout (t % every == 0): restoring force sum_a sum_r f^p(r) K(R_a - r) and the centre of
//     mass of R(t), FP64 sums in a fixed order; the last CTA also reduces the per-CTA partial sums
//     of the lattice kernel (mass, momentum, total force) in a fixed order;
//   * overdamped advection dR/dt = v(R) by Heun on the frozen u(t): R* = R + v(R),
//     R' = R + (v(R) + v(R*))/2, v interpolated with the cosine kernel (FP32 weights);
//   * Lagrangian forces of R' (Eq. Const: springs, angle terms, constant pull split over the
//     nodes), gathered per node without atomics, and the work box of R' for the next step.
// Node positions are kept in FP64 (O(N_nodes) data) and advanced in FP64; the forces are
// evaluated in FP32 except the spring extension, whose l^2 - l_eq^2 is formed in FP64.  The
// lattice kernel sees the nodes as int32 cell + FP32 fraction with FP32 forces.
//
// The node step of a small lattice is pure latency: it stands between the last tile of a step and
// the first gather of the next.  So one CTA advances a whole ring, with the edges exchanged through
// shared memory: three barriers, no partial results in global memory, no arrival counters between
// CTAs.  (Blocks of 60 nodes on CTAs of their own, with the ring's sums and box put together by the
// last of them, took 110 000 cycles for 157 nodes with the trap, 53 of the 74 us of a 250^2 step.)
#pragma once
#include <cuda_runtime.h>

#include "lb_cell.cuh"
#include "lb_internal.h"

namespace vlb {
namespace node {

// Node positions are kept in [0, n); one step moves a node by less than one cell, and offsets
// between nodes of a ring are below n/2, so single conditional corrections replace fmod.
__device__ __forceinline__ double wrap1(double x, double L)
{
    if (x < 0.0) x += L;
    else if (x >= L) x -= L;
    return x;
}

// d in (-L, L) to [-L/2, L/2); the comparisons on the bits (L/2 is L with its exponent one less)
// leave the FP64 pipe one subtraction where one is needed.
__device__ __forceinline__ double mimg1(double d, double L)
{
    const long long h = __double_as_longlong(L) - (1ll << 52), b = __double_as_longlong(d);
    if (b >= h) d -= L;
    else if (b < 0 && (b & 0x7fffffffffffffffll) > h) d += L;
    return d;
}

__device__ __forceinline__ int wrapi1(int i, int n)
{
    if (i < 0) i += n;
    else if (i >= n) i -= n;
    return i;
}

// The four cosine-kernel weights phi(f + 1), phi(f), phi(f - 1), phi(f - 2) of a node at
// fraction f in [0, 1) (App. A): with c = cos(pi f / 2), s = sin(pi f / 2) they are
// (1 - s)/4, (1 + c)/4, (1 + s)/4, (1 - c)/4 (quarter-period shifts of the cosine).
__device__ __forceinline__ void phi4(float f, float* w)
{
    float sn, cs;
    sincospif(0.5f * f, &sn, &cs);
    w[0] = 0.25f * (1.f - sn);
    w[1] = 0.25f * (1.f + cs);
    w[2] = 0.25f * (1.f + sn);
    w[3] = 0.25f * (1.f - cs);
}

// Cell and FP32 fraction of a coordinate x: (int)x and (float)(x - (int)x).  For x in [0, 2^20) the
// integer part is read off the bits (the masked double is it exactly), which leaves the FP64 pipe,
// one warp instruction in 16 cycles for the whole SM, one subtraction and one conversion.
__device__ __forceinline__ void cell_frac(double x, int& c, float& f)
{
    const int hi = __double2hiint(x), e = (hi >> 20) - 1023;
    if ((unsigned)hi < 0x41300000u) {
        const int sh = 20 - e;                               // 1 .. 20 for x >= 1
        const bool one = e >= 0;
        c = one ? ((hi & 0xfffff) | 0x100000) >> sh : 0;
        f = (float)(x - __hiloint2double(one ? hi & (-1 << sh) : 0, 0));
    } else {                                                 // negative, huge or NaN
        c = (int)x;
        f = (float)(x - c);
    }
}

// Interpolate one component of a box field for a node whose 4 x 4 cells start at p, in rows of
// `stride`: in global memory (written by the lattice step, so read through L2), or the box in
// shared memory (SM).
template <bool SM>
__device__ __forceinline__ float interp_sum(const float* p, int stride, const float* wx, const float* wy)
{
    float v = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float w = wx[i] * wy[j];
            v += w * (SM ? p[j * stride + i] : __ldcg(p + j * stride + i));
        }
    }
    return v;
}

// The same by a pair of lanes, the even one for x and the odd one for y: c in [0, n) and f are the
// node's cell and fraction on this lane's axis, (o, span) the box on that axis, ax the component;
// returns false in both lanes if a support cell lies outside the box.  The whole warp calls it.
__device__ __forceinline__ bool interp_pair(const float* box, int cap_w, long long cap, const float* staged, int box_w,
                                            int box_h, int ax, int n, int o, int c, float f, float& v)
{
    constexpr unsigned ALL = 0xffffffffu;
    int d = wrapi1(wrapi1(c - 1, n) - o, n);
    if (d < 0 || d + 3 >= (ax ? box_h : box_w)) d = -1;     // the box never wraps onto itself
    const int e = __shfl_xor_sync(ALL, d, 1);
    float w[4], wx[4], wy[4];
    phi4(f, w);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float u = __shfl_xor_sync(ALL, w[i], 1);
        wx[i] = ax ? u : w[i];
        wy[i] = ax ? w[i] : u;
    }
    const int ox = ax ? e : d, oy = ax ? d : e;
    v = 0.f;
    if (d < 0 || e < 0) return false;
    if (staged) v = interp_sum<true>(staged + (ax * box_h + oy) * box_w + ox, box_w, wx, wy);
    else v = interp_sum<false>(box + ax * cap + (long long)oy * cap_w + ox, cap_w, wx, wy);
    return true;
}

// The trap protocol at step t: k(t), and the trap's place x0 + dx g(t) with g the fraction of its way,
// from the sigmoids s(t; c) = 1 / (1 + exp(-8 (t - c) / w)) and softplus(z) = log(1 + e^z).  Two warps,
// half 0: k, half 1: the place; both points of time of each on a lane.  (Next to an FP64 instruction's
// 60 cycles for its warp: a division 580, exp 1 240, log1p 1 560.)
__device__ __forceinline__ void trap_at(const RingDev& R, double t, int half, double* out)
{
    const int lane = threadIdx.x & 31;
    const double w = R.trap_w, te = R.trap_t_eq, T = R.trap_pull;
    if (half == 0) {
        const double c = lane == 0 ? 0.5 * w : te + T + 0.5 * w;
        const double v = 1.0 / (1.0 + exp(-8.0 * (t - c) / w));
        const double s1 = __shfl_sync(0xffffffffu, v, 1);
        if (lane == 0) out[0] = R.trap_k * v * (1.0 - s1);
    } else {
        const double a = 8.0 / w;
        const double z = a * (lane == 0 ? t - te : t - te - T);
        const double l = log1p(exp(-fabs(z)));
        const double p = z > 0.0 ? z + l : l;
        const double p1 = __shfl_sync(0xffffffffu, p, 1);
        if (lane == 0) {
            const double g = (p - p1) / (a * T);
            out[1] = R.trap_x0 + R.trap_dx * g;
            out[2] = R.trap_y0 + R.trap_dy * g;
        }
    }
}

__device__ __forceinline__ int half_wrap(int d, int n)   // d in (-n, n) -> [-n/2, n/2)
{
    if (d >= n - n / 2) d -= n;
    else if (d < -(n / 2)) d += n;
    return d;
}

// Shared memory of one ring's node step.  It is passed in rather than declared static: a kernel
// that runs it after other work hands over space it no longer needs, so the node code takes
// nothing from the L1 share of that kernel's main work.  The pool holds, for a ring of n nodes, the
// new positions [n] double2, and behind them first u(t) on the ring's box (if it fits), then the
// edges: R_(k+1) - R_k [n] float2, tension / length [n] float and 1 / length [n] float.
struct NodeSmem {
    double2 pool[2 * MAX_RING_NODES];
    double sums[6][NODE_THREADS];                  // of the nodes k, k + NODE_THREADS, ...: F_rest, COM of
                                                   // R(t), COM of R(t+1)
    double dred[4 * 32];
    double trap[3];                                // k and the trap's place at the next step
    double leq2;
    float par[5];                                  // k_spring, eps_angle, l_eq, pull_x, pull_y
    int ext[4];                                    // cell extent: min x, -max x, min y, -max y
    int flag;                                      // free for the caller
    int s_last;
};
static_assert(sizeof(NodeSmem) <= 48 * 1024, "static shared memory of the node kernels");

// What the node step reads of a ring and, per thread, of its first node.  None of it is written
// during the step, so the tail of the lattice kernel loads it before it knows whether it is the
// last tile: one pass through L2 less in the chain.
struct RingRegs {
    int n, off, cap_w, cap_h;
    long long box_off;
    int4 B;
    bool trap;
    double X0;                   // thread 2 k + (0: x, 1: y): node k
};

__device__ __forceinline__ void load_first_node(const NodeArgs& a, RingRegs& q)
{
    q.X0 = 0.0;
    if ((int)threadIdx.x < 2 * q.n) q.X0 = reinterpret_cast<const double*>(a.X + q.off)[threadIdx.x];
}

__device__ __forceinline__ void load_ring(const NodeArgs& a, int ring, long long t, RingRegs& q)
{
    const RingDev& R = a.rings[ring];
    q.n = R.n_nodes;
    q.off = R.node_off;
    q.cap_w = R.cap_w;
    q.cap_h = R.cap_h;
    q.box_off = R.box_off;
    q.B = ring_box(R, t);
    q.trap = __double_as_longlong(R.trap_k) > 0;
}

// Lattice readout of step t, run by the last CTA to arrive (all its threads): the sums of the
// per-CTA partials (double-float pairs, cell::store_partial) in a fixed order, merged in
// double-float on FP32 lanes, into columns 0-5 of the readout row; FP64 only for the five totals.
// dred: 4 * 32 doubles of shared scratch.
__device__ __forceinline__ void lattice_readout(const NodeArgs& a, long long t, double* dred)
{
    const int tid = threadIdx.x;
    double* row = a.series + (long long)((t / a.every) % a.series_cap) * a.row_len;
    cell::DF v[5] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    // the partials of other CTAs, read through L2 (after the caller's fence), several in flight
    const float2* P = reinterpret_cast<const float2*>(a.partials);
#pragma unroll 4
    for (int k = tid; k < a.n_partials; k += blockDim.x) {
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            const float2 q = __ldcg(P + (long long)k * 5 + c);
            v[c] = cell::df_merge(v[c], cell::DF{q.x, q.y});
        }
    }
    const cell::DF s = cell::df_block_sum<5>(v, reinterpret_cast<float*>(dred));
    if (tid < 5) {
        const double val = (double)s.hi + (double)s.lo;
        row[1 + tid] = val;
        if (!isfinite(val)) atomicExch(&a.ctl->err_nonfinite, 1);
    }
    if (tid == 0) row[0] = (double)t;
}

// Sum of v[0 .. m) by a warp in a fixed order: a strided run per lane, a shuffle tree (lane 0).
__device__ __forceinline__ double warp_sum(const double* v, int m)
{
    double s = 0.0;
    for (int j = threadIdx.x & 31; j < m; j += 32) s += v[j];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;
}

// The node step of one ring by the whole CTA of NODE_THREADS threads; rg: load_ring and
// load_first_node, done.  Its time is latency and the FP64 pipe: an FP64 instruction holds its warp for
// 60 cycles whether it depends on the one before or not, and the SM takes one in 19.  So
//   * a pair of lanes advances a node, x and y: half the FP64 instructions, cosines and loads per warp;
//     cells come from the bits of a coordinate, comparisons are made on integers;
//   * u(t) on the box comes to shared memory in one coalesced pass (a lane per node read 2 x 32
//     scattered values, a wavefront each, twice);
//   * the trap's protocol, sums and force run on the last two warps beside everything else.
// A ring's step in the tail of a small lattice, cycles before and after: 32 nodes 15 700, 10 000; 157
// nodes with the trap 26 200, 19 700.
__device__ __forceinline__ void node_ring(const NodeArgs& a, int ring, const RingRegs& rg, NodeSmem& S, long long t,
                                          bool readout)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int NW = NODE_THREADS / 32;
    const int nx = a.nx, ny = a.ny;
    RingDev& R = a.rings[ring];
    const int n = rg.n, off = rg.off, cap_w = rg.cap_w;
    const long long cap = (long long)cap_w * rg.cap_h;
    const float* ubox = a.ubox + rg.box_off;
    const float* fpbox = a.fpbox + rg.box_off;
    const int4 B = rg.B;
    const bool trap = rg.trap;
    // the warps that advance nodes: without the last two where the trap keeps these busy, unless the
    // ring is so large that a thread's nodes have to be NODE_THREADS apart for the sums
    const int nwork = trap && n <= NODE_THREADS ? NODE_THREADS - 64 : NODE_THREADS;
    double* P = reinterpret_cast<double*>(S.pool);
    const double2* pos = S.pool;
    float* field = reinterpret_cast<float*>(S.pool + n);
    float2* edge = reinterpret_cast<float2*>(field);
    float* tens = reinterpret_cast<float*>(edge + n);
    float* ilen = tens + n;
    const float hx = 0.5f * (float)nx, hy = 0.5f * (float)ny;
    if (wid == NW - 3 && lane < 5) {
        const double p = lane == 0 ? R.k_spring : (lane == 1 ? R.eps_angle : (lane == 2 ? R.l_eq : (lane == 3 ? R.pull_x : R.pull_y)));
        S.par[lane] = (float)p;
        if (lane == 2) S.leq2 = p * p;
    }
    if (tid < 4) S.ext[tid] = 1 << 30;
    if (trap && wid >= NW - 2) trap_at(R, (double)(t + a.advance), wid - (NW - 2), S.trap);
    if (tid < nwork) {
        const float* staged = nullptr;
        if (a.advance && 8LL * B.z * B.w <= (long long)sizeof(S.pool) - 16 * n) {
            // u(t) on the box, rows of B.z, both components
            const int half = B.z * B.w, m = 2 * half;
            const float inv = 1.f / (float)B.z;
            for (int i0 = tid; i0 < m; i0 += 8 * nwork) {
                float v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = i0 + j * nwork;
                    const int c = i >= half, r = i - c * half;
                    const int y = (int)(((float)r + 0.5f) * inv);      // r / B.z: r < 2^13, half a cell off the edge
                    v[j] = i < m ? __ldcg(ubox + c * cap + (long long)y * cap_w + (r - y * B.z)) : 0.f;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (i0 + j * nwork < m) field[i0 + j * nwork] = v[j];
            }
            staged = field;
        }
        asm volatile("bar.sync 1, %0;" ::"r"(nwork) : "memory");
        // ---- advance: Heun on the frozen u(t); even lanes x, odd lanes y -----------------------
        const int ax = tid & 1, N = ax ? ny : nx, o = ax ? B.y : B.x;
        const float h = ax ? hy : hx;
        const bool wall = ax ? a.walls_y : a.walls_x;
        const double L = ax ? a.len_y : a.len_x, od = trap || readout ? (double)o : 0.0;
        bool bad = false;
        int mn = 1 << 30, mx = 1 << 30;                  // this lane's cell extent on its axis
        for (int base = 0; base + (tid & ~31) < 2 * n; base += nwork) {
            const int item = base + tid, k = min(item >> 1, n - 1);
            const bool act = item < 2 * n;               // as one for the two lanes of a pair
            const double X = base == 0 && act ? rg.X0 : reinterpret_cast<const double*>(a.X + off)[2 * k + ax];
            int c;
            float f;
            cell_frac(X, c, f);                          // X >= 0
            double Xn = X;
            if (a.advance) {
                const int kk = k & (NODE_THREADS - 1);
                if (readout) {
                    float p;
                    bad |= !interp_pair(fpbox, cap_w, cap, nullptr, B.z, B.w, ax, N, o, c, f, p);
                    const double q = mimg1(X - od, L);   // centre of mass relative to the box
                    if (act) {
                        S.sums[ax][kk] = k < NODE_THREADS ? (double)p : S.sums[ax][kk] + (double)p;
                        S.sums[2 + ax][kk] = k < NODE_THREADS ? q : S.sums[2 + ax][kk] + q;
                    }
                }
                float v, w;
                bad |= !interp_pair(ubox, cap_w, cap, staged, B.z, B.w, ax, N, o, c, f, v);
                // R* = R + v.  Moving by less than a cell, only a node in the lattice's outermost
                // cells can leave [0, n); beyond half the lattice (or NaN) there is no R*
                const bool rim = c == 0 || c >= N - 1;
                int ok = (fabsf(v) < h ? 1 : 0) | (fabsf(v) < 1.f ? 2 : 0);
                ok &= __shfl_xor_sync(0xffffffffu, ok, 1);
                const bool here = ok & 1;
                const double vd = v;
                double Xs = here ? X + vd : X;
                if (rim || !(ok & 2)) Xs = wrap1(Xs, L);
                int s;
                float g;
                cell_frac(Xs, s, g);
                bad |= !here;
                bad |= !interp_pair(ubox, cap_w, cap, staged, B.z, B.w, ax, N, o, s, g, w);
                // a node that moves by a cell or more in one step is an error
                int near = fabsf(0.5f * (v + w)) < 1.f;
                near &= __shfl_xor_sync(0xffffffffu, near, 1);
                bad |= !near;
                Xn = fma(0.5, vd + (double)w, X);
                if (rim || !near) Xn = wrap1(Xn, L);
                cell_frac(Xn, c, f);
                // supports stay off the walls: 4 <= Xn <= N - 5
                if (wall && (c < 4 || c > N - 5 || (c == N - 5 && f > 0.f))) bad = true;
            }
            if (act) P[2 * k + ax] = Xn;
            if (trap) {                                  // advanced positions, for the trap
                const int kk = k & (NODE_THREADS - 1);
                const double q = mimg1(Xn - od, L);
                if (act) S.sums[4 + ax][kk] = k < NODE_THREADS ? q : S.sums[4 + ax][kk] + q;
            }
            if (f >= 1.f) { f = 0.f; c += 1; }
            c = wrapi1(c, N);
            if (act) {
                reinterpret_cast<double*>(a.X_out + off)[item] = Xn;
                reinterpret_cast<int*>(a.node_cell + off)[item] = c;
                reinterpret_cast<float*>(a.node_frac + off)[item] = f;
            }
            // cell offsets from the previous box origin, for the new box
            const int u = half_wrap(c - o, N);
            mn = min(mn, u);
            mx = min(mx, -u);
        }
        if ((tid & ~31) < 2 * n) {
            const int m0 = __reduce_min_sync(0xffffffffu, ax ? 1 << 30 : mn), m1 = __reduce_min_sync(0xffffffffu, ax ? 1 << 30 : mx),
                      m2 = __reduce_min_sync(0xffffffffu, ax ? mn : 1 << 30), m3 = __reduce_min_sync(0xffffffffu, ax ? mx : 1 << 30);
            if (lane < 4) atomicMin(&S.ext[lane], lane == 0 ? m0 : (lane == 1 ? m1 : (lane == 2 ? m2 : m3)));
        }
        if (bad) atomicExch(&a.ctl->err_body, 1);
    }
    __syncthreads();
    // the staged field is dead from here on: the edges take its place
    if (trap && wid >= NW - 2) {
        // Eq. Utrap at the step the nodes advance to: k (R_ext - R_com) / N on each node, x and y on a
        // warp each
        const int c = wid - (NW - 2);
        const double v = warp_sum(S.sums[4 + c], min(n, NODE_THREADS));
        if (lane == 0) {
            const double e = mimg1(S.trap[1 + c] - ((double)(c == 0 ? B.x : B.y) + v / n), c == 0 ? a.len_x : a.len_y);
            reinterpret_cast<float*>(&R.trap_f[(t + a.advance) & 1])[c] = (float)(S.trap[0] * e / n);
        }
    }
    // the box of the step the nodes advance to: cells min-2 .. max+3
    if (tid == 32 * (NW - 3)) {
        int w = -S.ext[1] - S.ext[0] + 6, h = -S.ext[3] - S.ext[2] + 6;
        if (w > cap_w || h > rg.cap_h) {
            atomicExch(&a.ctl->err_body, 1);
            w = min(w, cap_w);
            h = min(h, rg.cap_h);
        }
        R.box[(t + a.advance) & 1] = make_int4(wrapi1(wrapi1(B.x + S.ext[0] - 2, nx), nx),
                                               wrapi1(wrapi1(B.y + S.ext[2] - 2, ny), ny), w, h);
    }
    // ---- edges: Eq. Const.  Spring on the edge (k, k+1): the extension l - l_eq = (l^2 -
    // l_eq^2) / (l + l_eq) with l^2 - l_eq^2 formed in FP64 from the FP64 edge vector, so it
    // keeps its relative precision; the rest in FP32.
    for (int k = tid; k < n; k += NODE_THREADS) {
        const double2 p0 = pos[k], p1 = pos[k + 1 == n ? 0 : k + 1];
        double qxd = p1.x - p0.x, qyd = p1.y - p0.y;
        float qx = (float)qxd, qy = (float)qyd;
        if (fabsf(qx) >= hx) {                           // across the seam
            qxd = mimg1(qxd, a.len_x);
            qx = (float)qxd;
        }
        if (fabsf(qy) >= hy) {
            qyd = mimg1(qyd, a.len_y);
            qy = (float)qyd;
        }
        const double ext2 = fma(qxd, qxd, fma(qyd, qyd, -S.leq2));
        const float l = sqrtf(qx * qx + qy * qy);
        edge[k] = make_float2(qx, qy);
        tens[k] = S.par[0] * (float)ext2 / ((l + S.par[2]) * l);
        ilen[k] = 1.f / l;
    }
    __syncthreads();
    // ---- forces: f_a = -dU/dR_a: springs (a, a+1) and (a-1, a); angle terms at a-1 (a is its
    // next), a, a+1 (a is its prev); the pull
    for (int k = tid; k < n; k += NODE_THREADS) {
        // gradients of cos(gamma_j) = p.q / (|p||q|) at j, p = R_(j-1) - R_j, q = R_(j+1) - R_j
        auto angle = [&](int j, float2& dp, float2& dq) {
            const int jm = j == 0 ? n - 1 : j - 1;
            const float2 q = edge[j], e = edge[jm];
            const float iq = ilen[j], ip = ilen[jm];
            const float2 p = make_float2(-e.x, -e.y);
            const float ipq = ip * iq;
            const float c = (p.x * q.x + p.y * q.y) * ipq;
            const float cp = c * ip * ip, cq = c * iq * iq;
            dp = make_float2(q.x * ipq - cp * p.x, q.y * ipq - cp * p.y);
            dq = make_float2(p.x * ipq - cq * q.x, p.y * ipq - cq * q.y);
        };
        const int km = k == 0 ? n - 1 : k - 1, kp = k + 1 == n ? 0 : k + 1;
        float2 dpm, dqm, dp0, dq0, dpp, dqp;
        angle(km, dpm, dqm);
        angle(k, dp0, dq0);
        angle(kp, dpp, dqp);
        const float2 q0 = edge[k], qm = edge[km];
        const float T0 = tens[k], Tm = tens[km], eps = S.par[1];
        const float fx = T0 * q0.x - Tm * qm.x - eps * (dpp.x + dqm.x - dp0.x - dq0.x) + S.par[3];
        const float fy = T0 * q0.y - Tm * qm.y - eps * (dpp.y + dqm.y - dp0.y - dq0.y) + S.par[4];
        a.node_force[off + k] = make_float2(fx, fy);
        if (!isfinite(fx) || !isfinite(fy)) atomicExch(&a.ctl->err_nonfinite, 1);
    }
    if (readout && wid < 4) {
        const double v = warp_sum(S.sums[wid], min(n, NODE_THREADS));
        if (lane == 0) {
            double* rr = a.series + (long long)((t / a.every) % a.series_cap) * a.row_len + 6 + 4 * ring;
            rr[wid] = wid < 2 ? v : (wid == 2 ? wrap1((double)B.x + v / n, a.len_x) : wrap1((double)B.y + v / n, a.len_y));
            if (!isfinite(v)) atomicExch(&a.ctl->err_nonfinite, 1);
        }
    }
}

// A node launch's CTA (k_nodes, the batched kernels): one ring (-1: none), then, by the last CTA
// overall, the end of the step.
__device__ __forceinline__ void node_step(const NodeArgs& a, int ring, NodeSmem& S)
{
    const int tid = threadIdx.x;
    const long long t = a.ctl->t;
    const bool readout = a.advance && (t % a.every) == 0;
    RingRegs q;
    if (ring >= 0) load_ring(a, ring, t, q);
    // u(t), f^p(t) and the lattice readout sums come from the lattice kernel just before
    cell::pdl_wait();
    cell::pdl_trigger();
    if (ring >= 0) {
        load_first_node(a, q);
        node_ring(a, ring, q, S, t, readout);
    }
    // the last CTA overall: lattice readout sums (fixed order) and the step counter
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&a.ctl->ticket, 1u);
        S.s_last = (prev == (unsigned)a.n_ctas - 1u);
    }
    __syncthreads();
    if (S.s_last) {
        __threadfence();
        if (readout) lattice_readout(a, t, S.dred);
        if (tid == 0) {
            a.ctl->ticket = 0u;
            if (a.advance) a.ctl->t = t + a.advance;      // advance: steps taken (1, or a jump)
            __threadfence();
        }
    }
}

}  // namespace node
}  // namespace vlb
