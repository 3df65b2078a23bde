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
// the first gather of the next.  So one CTA advances a whole ring (thread k the nodes k, k + 256,
// ...), with the edges exchanged through shared memory: three barriers, no partial results in
// global memory, no arrival counters between CTAs.  Blocks of 60 nodes on CTAs of their own, with
// the ring's sums and box put together by the last of them, took 27 000 cycles a block (157 nodes
// and the trap: 110 000 cycles, 53 of the 74 us of a 250^2 step).  FP64 instructions occupy the SM's FP64
// pipe for 16 cycles each, so cells and offsets are integers and FP32 wherever they are exact.
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

__device__ __forceinline__ double mimg1(double d, double L)
{
    if (d >= 0.5 * L) d -= L;
    else if (d < -0.5 * L) d += L;
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

// Interpolate a 2-component box field for a node at cell (cx, cy) in [0, n) with fractions
// (fx, fy); returns false if a support cell lies outside the box.
__device__ __forceinline__ bool interp_box(const float* box, int cap_w, long long cap, const int4& B, int nx, int ny,
                                           int cx, int cy, float fx, float fy, float& vx, float& vy)
{
    const int ox = wrapi1(wrapi1(cx - 1, nx) - B.x, nx), oy = wrapi1(wrapi1(cy - 1, ny) - B.y, ny);
    vx = 0.f;
    vy = 0.f;
    if (ox < 0 || oy < 0 || ox + 3 >= B.z || oy + 3 >= B.w) return false;   // the box never wraps onto itself
    float wx[4], wy[4];
    phi4(fx, wx);
    phi4(fy, wy);
    const float* p = box + (long long)oy * cap_w + ox;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float w = wx[i] * wy[j];
            vx += w * __ldcg(p + j * cap_w + i);        // written by the lattice step
            vy += w * __ldcg(p + j * cap_w + i + cap);
        }
    }
    return true;
}

// The trap protocol at step t (doubles): k(t) and the trap's fraction g(t) of its way, from the
// sigmoids s(t; c) = 1 / (1 + exp(-8 (t - c) / w)).
__device__ __forceinline__ double trap_sigmoid(double t, double c, double w) { return 1.0 / (1.0 + exp(-8.0 * (t - c) / w)); }
__device__ __forceinline__ double trap_softplus(double z) { return z > 0.0 ? z + log1p(exp(-z)) : log1p(exp(z)); }
// k(t) and g(t) by four lanes at once (lanes 0, 1: the two sigmoids; 2, 3: the two softplus), valid
// in lane 0; the whole warp calls it.
__device__ __forceinline__ void trap_at(const RingDev& R, double t, double& k, double& g)
{
    const int lane = threadIdx.x & 31;
    const double w = R.trap_w, te = R.trap_t_eq, T = R.trap_pull;
    const double a = 8.0 / w;
    double v = 0.0;
    if (lane < 2) v = trap_sigmoid(t, lane == 0 ? 0.5 * w : te + T + 0.5 * w, w);
    else if (lane < 4) v = trap_softplus(a * (lane == 2 ? t - te : t - te - T));
    const double s1 = __shfl_sync(0xffffffffu, v, 1), p0 = __shfl_sync(0xffffffffu, v, 2),
                 p1 = __shfl_sync(0xffffffffu, v, 3);
    k = R.trap_k * v * (1.0 - s1);
    g = (p0 - p1) / (a * T);
}

__device__ __forceinline__ int half_wrap(int d, int n)   // d in (-n, n) -> [-n/2, n/2)
{
    if (d >= n - n / 2) d -= n;
    else if (d < -(n / 2)) d += n;
    return d;
}

// Shared memory of one ring's node step.  It is passed in rather than declared static: a kernel
// that runs it after other work hands over space it no longer needs, so the node code takes
// nothing from the L1 share of that kernel's main work.
struct NodeSmem {
    double2 pos[MAX_RING_NODES];                   // new positions; later the threads' sums
    float2 edge[MAX_RING_NODES];                   // R_(k+1) - R_k
    float2 tens[MAX_RING_NODES];                   // spring tension vector of that edge
    float ilen[MAX_RING_NODES];                    // 1 / its length
    double dred[4 * 32];
    double trap[2];                                // k(t), g(t) of the next step
    int ext[4];                                    // cell extent: min x, -max x, min y, -max y
    int flag;                                      // free for the caller
    int s_last;
};
static_assert(6 * NODE_THREADS * sizeof(double) <= MAX_RING_NODES * sizeof(double2), "sums overlay the positions");

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

// The node step of one ring (-1: none) by the whole CTA of NODE_THREADS threads; called by k_nodes
// and the batched kernels (one ring per CTA) and (whole_step = false: without the end of the step,
// which the caller then runs itself; t_in: the step index, else read from ctl->t) by the tail of
// the lattice kernel.
__device__ __forceinline__ void node_ring(const NodeArgs& a, int ring, NodeSmem& S, bool whole_step = true,
                                          long long t_in = -1)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nx = a.nx, ny = a.ny;
    const double Lx = nx, Ly = ny;
    const long long t = t_in >= 0 ? t_in : a.ctl->t;
    const bool readout = a.advance && (t % a.every) == 0;

    if (ring >= 0) {
        RingDev& R = a.rings[ring];
        const int n = R.n_nodes, off = R.node_off, cap_w = R.cap_w;
        const long long cap = (long long)cap_w * R.cap_h;
        const float* ubox = a.ubox + R.box_off;
        const float* fpbox = a.fpbox + R.box_off;
        const int4 B = ring_box(R, t);
        const bool trap = R.trap_k > 0.0;
        double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};     // F_rest, COM of R(t), COM of R(t+1)
        bool bad = false;
        int m0 = 1 << 30, m1 = 1 << 30, m2 = 1 << 30, m3 = 1 << 30;   // this thread's cell extent
        const float hx = 0.5f * (float)nx, hy = 0.5f * (float)ny;
        if (tid < 4) S.ext[tid] = 1 << 30;
        // u(t), f^p(t) and the lattice readout sums come from the lattice kernel just before
        cell::pdl_wait();
        cell::pdl_trigger();
        __syncthreads();
        if (trap && wid == NODE_THREADS / 32 - 1) {         // a warp that holds no node of most rings
            double kt, g;
            trap_at(R, (double)(t + a.advance), kt, g);
            if (lane == 0) {
                S.trap[0] = kt;
                S.trap[1] = g;
            }
        }
        // ---- advance: Heun on the frozen u(t) --------------------------------------------------
        for (int k = tid; k < n; k += NODE_THREADS) {
            const double2 X = a.X[off + k];
            int cx = (int)X.x, cy = (int)X.y;               // X, Y >= 0
            float fx = (float)(X.x - cx), fy = (float)(X.y - cy);
            double2 Xn = X;
            if (a.advance) {
                if (readout) {
                    float px, py;
                    bad |= !interp_box(fpbox, cap_w, cap, B, nx, ny, cx, cy, fx, fy, px, py);
                    acc[0] += (double)px;
                    acc[1] += (double)py;
                    acc[2] += mimg1(X.x - (double)B.x, Lx);       // centre of mass relative to the box
                    acc[3] += mimg1(X.y - (double)B.y, Ly);
                }
                float vx, vy, wx, wy;
                bad |= !interp_box(ubox, cap_w, cap, B, nx, ny, cx, cy, fx, fy, vx, vy);
                // R* = R + v.  Moving by less than a cell, only a node in the lattice's outermost
                // cells can leave [0, n); beyond half the lattice (or NaN) there is no R*
                const bool edge_x = cx == 0 || cx >= nx - 1, edge_y = cy == 0 || cy >= ny - 1;
                const bool here = fabsf(vx) < hx && fabsf(vy) < hy;
                const bool far0 = !(fabsf(vx) < 1.f && fabsf(vy) < 1.f);
                double Xs = X.x + (double)(here ? vx : 0.f), Ys = X.y + (double)(here ? vy : 0.f);
                if (edge_x || far0) Xs = wrap1(Xs, Lx);
                if (edge_y || far0) Ys = wrap1(Ys, Ly);
                const int sx = (int)Xs, sy = (int)Ys;
                bad |= !here;
                bad |= !interp_box(ubox, cap_w, cap, B, nx, ny, sx, sy, (float)(Xs - sx), (float)(Ys - sy), wx, wy);
                // a node that moves by a cell or more in one step is an error
                const bool far = !(fabsf(0.5f * (vx + wx)) < 1.f && fabsf(0.5f * (vy + wy)) < 1.f);
                bad |= far;
                Xn.x = fma(0.5, (double)vx + (double)wx, X.x);
                Xn.y = fma(0.5, (double)vy + (double)wy, X.y);
                if (edge_x || far) Xn.x = wrap1(Xn.x, Lx);
                if (edge_y || far) Xn.y = wrap1(Xn.y, Ly);
                if (a.walls_y && (Xn.y < 4.0 || Xn.y > Ly - 5.0)) bad = true;   // supports stay off the walls
                if (a.walls_x && (Xn.x < 4.0 || Xn.x > Lx - 5.0)) bad = true;
                cx = (int)Xn.x;
                cy = (int)Xn.y;
                fx = (float)(Xn.x - cx);
                fy = (float)(Xn.y - cy);
            }
            S.pos[k] = Xn;
            if (trap) {                                      // advanced positions, for the trap
                acc[4] += mimg1(Xn.x - (double)B.x, Lx);
                acc[5] += mimg1(Xn.y - (double)B.y, Ly);
            }
            a.X_out[off + k] = Xn;
            if (fx >= 1.f) { fx = 0.f; cx += 1; }
            if (fy >= 1.f) { fy = 0.f; cy += 1; }
            cx = wrapi1(cx, nx);
            cy = wrapi1(cy, ny);
            a.node_cell[off + k] = make_int2(cx, cy);
            a.node_frac[off + k] = make_float2(fx, fy);
            // cell offsets from the previous box origin, for the new box
            const int ux = half_wrap(cx - B.x, nx), uy = half_wrap(cy - B.y, ny);
            m0 = min(m0, ux);
            m1 = min(m1, -ux);
            m2 = min(m2, uy);
            m3 = min(m3, -uy);
        }
        m0 = __reduce_min_sync(0xffffffffu, m0);
        m1 = __reduce_min_sync(0xffffffffu, m1);
        m2 = __reduce_min_sync(0xffffffffu, m2);
        m3 = __reduce_min_sync(0xffffffffu, m3);
        if (lane < 4 && wid * 32 < n) atomicMin(&S.ext[lane], lane == 0 ? m0 : (lane == 1 ? m1 : (lane == 2 ? m2 : m3)));
        if (bad) atomicExch(&a.ctl->err_body, 1);
        __syncthreads();
        // ---- edges: Eq. Const.  Spring on the edge (k, k+1): the extension l - l_eq = (l^2 -
        // l_eq^2) / (l + l_eq) with l^2 - l_eq^2 formed in FP64 from the FP64 edge vector, so it
        // keeps its relative precision; the rest in FP32.
        const float ks = (float)R.k_spring, leq = (float)R.l_eq, eps = (float)R.eps_angle;
        const double leq2 = R.l_eq * R.l_eq;
        for (int k = tid; k < n; k += NODE_THREADS) {
            const double2 p0 = S.pos[k], p1 = S.pos[k + 1 == n ? 0 : k + 1];
            double qxd = p1.x - p0.x, qyd = p1.y - p0.y;
            if (fabsf((float)qxd) >= hx) qxd = mimg1(qxd, Lx);   // across the seam
            if (fabsf((float)qyd) >= hy) qyd = mimg1(qyd, Ly);
            const double ext2 = fma(qxd, qxd, fma(qyd, qyd, -leq2));
            const float qx = (float)qxd, qy = (float)qyd;
            const float l = sqrtf(qx * qx + qy * qy);
            const float T = ks * (float)ext2 / ((l + leq) * l);
            S.edge[k] = make_float2(qx, qy);
            S.tens[k] = make_float2(T * qx, T * qy);
            S.ilen[k] = 1.f / l;
        }
        __syncthreads();
        // ---- forces: f_a = -dU/dR_a: springs (a, a+1) and (a-1, a); angle terms at a-1 (a is its
        // next), a, a+1 (a is its prev); the pull
        for (int k = tid; k < n; k += NODE_THREADS) {
            // gradients of cos(gamma_j) = p.q / (|p||q|) at j, p = R_(j-1) - R_j, q = R_(j+1) - R_j
            auto angle = [&](int j, float2& dp, float2& dq) {
                const int jm = j == 0 ? n - 1 : j - 1;
                const float2 q = S.edge[j], e = S.edge[jm];
                const float iq = S.ilen[j], ip = S.ilen[jm];
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
            const float2 t0 = S.tens[k], tm = S.tens[km];
            const float fx = t0.x - tm.x - eps * (dpp.x + dqm.x - dp0.x - dq0.x) + (float)R.pull_x;
            const float fy = t0.y - tm.y - eps * (dpp.y + dqm.y - dp0.y - dq0.y) + (float)R.pull_y;
            a.node_force[off + k] = make_float2(fx, fy);
            if (!isfinite(fx) || !isfinite(fy)) atomicExch(&a.ctl->err_nonfinite, 1);
        }
        // the box of the step the nodes advance to: cells min-2 .. max+3
        if (tid == 0) {
            int w = -S.ext[1] - S.ext[0] + 6, h = -S.ext[3] - S.ext[2] + 6;
            if (w > cap_w || h > R.cap_h) {
                atomicExch(&a.ctl->err_body, 1);
                w = min(w, cap_w);
                h = min(h, R.cap_h);
            }
            R.box[(t + a.advance) & 1] = make_int4(wrapi1(wrapi1(B.x + S.ext[0] - 2, nx), nx),
                                                   wrapi1(wrapi1(B.y + S.ext[2] - 2, ny), ny), w, h);
        }
        if (readout || trap) {
            // fixed-order FP64 sums: each thread's nodes in order, then warp c < 6 adds value c (a
            // strided run per lane, a shuffle tree)
            double* sum = reinterpret_cast<double*>(S.pos);  // the positions were last read before the barrier
#pragma unroll
            for (int c = 0; c < 6; ++c) sum[c * NODE_THREADS + tid] = acc[c];
            __syncthreads();
            double v = 0.0;
            if (wid < 6 && (readout || wid >= 4)) {
                const int m = min(n, NODE_THREADS);
                for (int j = lane; j < m; j += 32) v += sum[wid * NODE_THREADS + j];
                for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            }
            if (lane == 0 && wid < 6) S.dred[wid] = v;
            __syncthreads();
            if (tid == 0 && trap) {
                // Eq. Utrap at the step the nodes advance to: k (R_ext - R_com) / N on each node
                const double kt = S.trap[0], g = S.trap[1];
                const double ex = mimg1(R.trap_x0 + R.trap_dx * g - ((double)B.x + S.dred[4] / n), Lx);
                const double ey = mimg1(R.trap_y0 + R.trap_dy * g - ((double)B.y + S.dred[5] / n), Ly);
                R.trap_f[(t + a.advance) & 1] = make_float2((float)(kt * ex / n), (float)(kt * ey / n));
            }
            if (readout && tid >= 32 && tid < 36) {
                const int c = tid - 32;
                double* rr = a.series + (long long)((t / a.every) % a.series_cap) * a.row_len + 6 + 4 * ring;
                const double s = S.dred[c];
                rr[c] = c < 2 ? s : (c == 2 ? wrap1((double)B.x + s / n, Lx) : wrap1((double)B.y + s / n, Ly));
                if (!isfinite(s)) atomicExch(&a.ctl->err_nonfinite, 1);
            }
        }
    }

    if (!whole_step) return;
    // the last CTA overall: lattice readout sums (fixed order) and the step counter
    if (ring < 0) {
        cell::pdl_wait();
        cell::pdl_trigger();
    }
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
