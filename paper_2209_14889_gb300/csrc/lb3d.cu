// lb3d.cu -- the three-dimensional form of the step (include/lb3d.h): D3Q19 lattice Boltzmann
// with the Guo force, the polymer stress of Eq. StiffCons with the stiffness averaged over the
// unit sphere, and the Beris-Edwards field P, as four HBM-streaming stencil kernels per step.
//
// Kernels of one step (one thread per cell, CTAs of 32 x 4 x 2 cells, x fastest so that a warp
// reads 128 contiguous bytes of a plane; neighbour values come through L1/L2):
//   k3_molecular  sigma^E (Sec. II C 1) of the state, from h = (alpha + beta |P|^2) P - kappa lap P
//                 (launched with the Ericksen force only)
//   k3_collide    F = div sigma^p + div sigma^E + f_ext, moments with the Guo half force, BGK
//                 collision with the Guo source pushed to the neighbours (Eq. LB, Eq. BGK); u;
//                 on readout steps the FP64 sums (mass, momentum, force) in a fixed order
//   k3_predict    RHS(y) of Eq. StiffCons and Eq. BE at y = (sigma^p, P) (h from the P stencils it
//                 loads), u(t) frozen; y* = y + RHS
//   k3_correct    RHS(y*) (h* from P*), y' = y + (RHS(y) + RHS(y*)) / 2 into the next state
// The stiffness C(P) = int g(n) K(n) dOmega is applied in its transversely isotropic form about
// P^: with the orientation moments m2 = <mu^2>, m4 = <mu^4> of the Fisher density (their
// combinations below tabulated against |P| in FP64 and stored as FP32),
// M2 = <nn> = A d + B pp and M4 = <nnnn> = e1 pppp + e2 Sym(pp d) + e3 Sym(d d), and
// K(n) = a1 nnnn + a2 (nn d + d nn) + a3 d d + a4 Sym'(nn d) + a5 (d d + d d), the contraction
// C:X of a symmetric X is
//   c_pp pp + c_d d + c_s (p (Xp) + (Xp) p) + c_X X
// with c_pp = a1 e1 pXp + (a1 e2 + a2 B) trX, c_d = (a1 e2 + a2 B) pXp + (a1 e3 + 2 a2 A + a3) trX,
// c_s = 2 (a1 e2 + a4 B), c_X = 2 (a1 e3 + 2 a4 A + a5).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/lb3d.h"
#include "lb_device_ptr.h"
#include "lb_vec.cuh"

namespace v3 {

constexpr int NQ = 19;
constexpr int NPL = 28;                 // 19 populations, 6 sigma, 3 P
constexpr int PL_S = 19, PL_P = 25;
constexpr int LUT_N = 8192;             // table intervals in |P| up to P_cap (linear interpolation:
                                        // coefficient error below 1e-7 of their scale)
constexpr int BX = 32, BY = 4, BZ = 2, NT = BX * BY * BZ;

// D3Q19 (the order of include/lb3d.h)
__device__ constexpr int CX[NQ] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
__device__ constexpr int CY[NQ] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
__device__ constexpr int CZ[NQ] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};

__device__ __forceinline__ float wq(int n) { return n == 0 ? 1.f / 3.f : (n < 7 ? 1.f / 18.f : 1.f / 36.f); }

struct Args3 {
    const float* src;            // state at t (NPL planes)
    float* dst;                  // state at t + 1
    float* sE;                   // Ericksen stress [9] (i * 3 + j)
    float* u;                    // u(t) [3]
    float* ys;                   // predictor y* [9]
    float* r0;                   // RHS(y) [9]
    const float4* lut;           // coefficients of C:X against |P| (two float4 per entry)
    long long NP;
    int nx, ny, nz;
    float tau_inv, guo, rho0;
    float inv_eta, Dp, alpha, beta, xi, Gamma, kappa, P_cap, lut_scale;
    float fx, fy, fz;
    float prx, pry, prz, A0;     // P_ref and alpha + beta |P_ref|^2 (formed in FP64)
    int ericksen;
    int readout;                 // k3_collide: sum the readouts of this step
    long long t;
    unsigned n_ctas;             // CTAs of k3_collide
    long long ahead;             // cells ahead whose planes the stencil kernels prefetch into L2 (0: none)
    double* partials;            // [n_ctas][7]
    double* gpartials;           // [groups of NT CTAs][7]
    double* row;                 // readout row of this step (8 values)
    int* err_nonfinite;
};

struct Cell {
    int x, y, z, c;
    int xp, xm, yp, ym, zp, zm;  // flat indices of the six face neighbours
};

__device__ __forceinline__ bool cell_of(const Args3& a, Cell& q)
{
    q.x = blockIdx.x * BX + threadIdx.x;
    q.y = blockIdx.y * BY + threadIdx.y;
    q.z = blockIdx.z * BZ + threadIdx.z;
    if (q.x >= a.nx || q.y >= a.ny || q.z >= a.nz) return false;
    const int nx = a.nx, nxy = a.nx * a.ny;
    q.c = q.z * nxy + q.y * nx + q.x;
    // neighbour offsets compose: the +x neighbour of the +y neighbour is c + (xp - c) + (yp - c)
    q.xp = q.c + (q.x + 1 == nx ? 1 - nx : 1);
    q.xm = q.c + (q.x == 0 ? nx - 1 : -1);
    q.yp = q.c + (q.y + 1 == a.ny ? nx - nxy : nx);
    q.ym = q.c + (q.y == 0 ? nxy - nx : -nx);
    q.zp = q.c + (q.z + 1 == a.nz ? nxy - nxy * a.nz : nxy);
    q.zm = q.c + (q.z == 0 ? nxy * a.nz - nxy : -nxy);
    return true;
}

// value of plane f at the cell and its six neighbours: v[0] centre, then +x -x +y -y +z -z
__device__ __forceinline__ void stencil(const float* f, const Cell& q, float* v)
{
    v[0] = f[q.c];
    v[1] = f[q.xp]; v[2] = f[q.xm];
    v[3] = f[q.yp]; v[4] = f[q.ym];
    v[5] = f[q.zp]; v[6] = f[q.zm];
}

__device__ __forceinline__ float lap7(const float* v) { return v[1] + v[2] + v[3] + v[4] + v[5] + v[6] - 6.f * v[0]; }
__device__ __forceinline__ float dif(const float* v, int a) { return 0.5f * (v[1 + 2 * a] - v[2 + 2 * a]); }

// alpha + beta |P|^2 at P = P_ref + dP without the cancellation near the equilibrium modulus
template <class T>
__device__ __forceinline__ T bulk(const Args3& a, T dx, T dy, T dz)
{
    using vlb::vec::vfma;
    using vlb::vec::operator*;
    const T pd = vfma(a.prx, dx, vfma(a.pry, dy, a.prz * dz));
    const T dd = vfma(dx, dx, vfma(dy, dy, dz * dz));
    return vfma(a.beta, vfma(2.f, pd, dd), vlb::vec::bc<T>(a.A0));
}

// symmetric-tensor component (xx, yy, zz, yz, xz, xy) of (i, j)
__device__ __forceinline__ int sym6(int i, int j)
{
    return i == j ? i : (i + j == 3 ? 3 : (i + j == 2 ? 4 : 5));
}

// One cell per thread (T = float) or the two cells x, x + 1 (T = float2, x even: nx even), whose
// arithmetic then runs on paired FP32 instructions and whose stencil points other than +-x are 8-byte
// loads.
using vlb::vec::operator+;
using vlb::vec::operator-;
using vlb::vec::operator*;
using vlb::vec::bc;
using vlb::vec::vfma;

// Consecutive kernels of a step overlap by programmatic dependent launch: each waits for the one before
// it to complete before it touches memory, then lets the next one start its CTAs.  What the kernels before
// have written is read by plain loads: the read-only path (__ldg) is for data that nothing writes while the
// kernel lives, and this kernel lives before the former one has ended; a compiler may also move such a load
// above the wait.  Only the coefficient table is read through it.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class T>
struct Nb {                      // flat indices: the cell (pair), +x of its last cell, -x of its first, +-y, +-z
    int c, xp, xm, yp, ym, zp, zm;
};

template <class T>
__device__ __forceinline__ bool nb_of(const Args3& a, Nb<T>& q)
{
    constexpr int W = vlb::vec::Lanes<T>::N;
    const int x = W * (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y * blockDim.y + threadIdx.y, z = blockIdx.z * blockDim.z + threadIdx.z;
    if (x >= a.nx || y >= a.ny || z >= a.nz) return false;
    const int nx = a.nx, nxy = a.nx * a.ny;
    q.c = z * nxy + y * nx + x;
    q.xp = q.c + (x + W == nx ? W - nx : W);
    q.xm = q.c + (x == 0 ? nx - 1 : -1);
    q.yp = q.c + (y + 1 == a.ny ? nx - nxy : nx);
    q.ym = q.c + (y == 0 ? nxy - nx : -nx);
    q.zp = q.c + (z + 1 == a.nz ? nxy - nxy * a.nz : nxy);
    q.zm = q.c + (z == 0 ? nxy * a.nz - nxy : -nxy);
    return true;
}

// The stencil kernels' loads, in program order behind the wait (256^3: 1758 us per step as with __ldg, where
// loads that the compiler may move spill registers and take 1777).
__device__ __forceinline__ float ldo(const float* p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
template <class T>
__device__ __forceinline__ T ldv(const float* p);
template <>
__device__ __forceinline__ float ldv<float>(const float* p) { return ldo(p); }
template <>
__device__ __forceinline__ float2 ldv<float2>(const float* p)
{
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
template <class T>
__device__ __forceinline__ void stv(float* p, T v) { *reinterpret_cast<T*>(p) = v; }

// value, differences f(+) - f(-) along x, y, z and the sum of the six neighbours of plane f
__device__ __forceinline__ void fold(const float* f, const Nb<float>& q, float& c, float& dx, float& dy, float& dz, float& sum)
{
    c = ldo(f + q.c);
    const float xp = ldo(f + q.xp), xm = ldo(f + q.xm), yp = ldo(f + q.yp), ym = ldo(f + q.ym),
                zp = ldo(f + q.zp), zm = ldo(f + q.zm);
    dx = xp - xm;
    dy = yp - ym;
    dz = zp - zm;
    sum = ((xp + xm) + (yp + ym)) + (zp + zm);
}
__device__ __forceinline__ void fold(const float* f, const Nb<float2>& q, float2& c, float2& dx, float2& dy, float2& dz,
                                     float2& sum)
{
    c = ldv<float2>(f + q.c);
    const float r = ldo(f + q.xp), l = ldo(f + q.xm);
    const float2 yp = ldv<float2>(f + q.yp), ym = ldv<float2>(f + q.ym), zp = ldv<float2>(f + q.zp), zm = ldv<float2>(f + q.zm);
    const float2 xp = make_float2(c.y, r), xm = make_float2(l, c.x);
    dx = xp - xm;
    dy = yp - ym;
    dz = zp - zm;
    sum = ((xp + xm) + (yp + ym)) + (zp + zm);
}

// ---- stiffness: the transversely isotropic contraction C(P):X --------------------------------
template <class T>
struct Stiff {
    T n[3];
    T cpp_n, g;                  // c_pp = cpp_n pXp + g trX
    T cd_t;                      // c_d  = g pXp + cd_t trX
    T cs, cX;
};

// The table holds, per |P|, the five scalar coefficients of C:X (formed on the host in FP64 from
// the orientation moments and K^x, so the cancellations in e1, e2, e3 never happen in FP32):
// (cpp_n, g, cd_t, cs) and (cX, -, -, -).
__device__ __forceinline__ void stiffness(const Args3& a, const float (&p)[3], Stiff<float>& S)
{
    const float Pm = sqrtf(p[0] * p[0] + p[1] * p[1] + p[2] * p[2]);
    if (Pm > 0.f) {
        const float r = 1.f / Pm;
        S.n[0] = p[0] * r; S.n[1] = p[1] * r; S.n[2] = p[2] * r;
    } else {
        S.n[0] = 1.f; S.n[1] = 0.f; S.n[2] = 0.f;
    }
    const float q = fminf(Pm, a.P_cap) * a.lut_scale;
    int i = (int)q;
    if (i > LUT_N - 1) i = LUT_N - 1;
    const float f = q - (float)i;
    const float4 u0 = __ldg(a.lut + 2 * i), u1 = __ldg(a.lut + 2 * i + 2);
    const float v0 = __ldg(&a.lut[2 * i + 1].x), v1 = __ldg(&a.lut[2 * i + 3].x);
    S.cpp_n = u0.x + f * (u1.x - u0.x);
    S.g = u0.y + f * (u1.y - u0.y);
    S.cd_t = u0.z + f * (u1.z - u0.z);
    S.cs = u0.w + f * (u1.w - u0.w);
    S.cX = v0 + f * (v1 - v0);
}
__device__ __forceinline__ void stiffness(const Args3& a, const float2 (&p)[3], Stiff<float2>& S)
{
    Stiff<float> A, B;
    const float pa[3] = {p[0].x, p[1].x, p[2].x}, pb[3] = {p[0].y, p[1].y, p[2].y};
    stiffness(a, pa, A);
    stiffness(a, pb, B);
#pragma unroll
    for (int i = 0; i < 3; ++i) S.n[i] = make_float2(A.n[i], B.n[i]);
    S.cpp_n = make_float2(A.cpp_n, B.cpp_n);
    S.g = make_float2(A.g, B.g);
    S.cd_t = make_float2(A.cd_t, B.cd_t);
    S.cs = make_float2(A.cs, B.cs);
    S.cX = make_float2(A.cX, B.cX);
}

// out = C:X for the symmetric X (6 components)
template <class T>
__device__ __forceinline__ void apply_c(const Stiff<T>& S, const T* X, T* out)
{
    const T* n = S.n;
    const T Xn[3] = {vfma(X[0], n[0], vfma(X[5], n[1], X[4] * n[2])), vfma(X[5], n[0], vfma(X[1], n[1], X[3] * n[2])),
                     vfma(X[4], n[0], vfma(X[3], n[1], X[2] * n[2]))};
    const T nXn = vfma(n[0], Xn[0], vfma(n[1], Xn[1], n[2] * Xn[2]));
    const T tr = (X[0] + X[1]) + X[2];
    const T cpp = vfma(S.cpp_n, nXn, S.g * tr);
    const T cd = vfma(S.g, nXn, S.cd_t * tr);
    // cpp n_i n_j + cs (n_i Xn_j + Xn_i n_j) = n_i V_j + V_i n_j with V = cpp n / 2 + cs Xn
    const T hc = 0.5f * cpp;
    T V[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) V[i] = vfma(hc, n[i], S.cs * Xn[i]);
    const int I[6] = {0, 1, 2, 1, 0, 0}, J[6] = {0, 1, 2, 2, 2, 1};
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const int i = I[c], j = J[c];
        if (i == j) out[c] = vfma(2.f * n[i], V[i], vfma(S.cX, X[c], cd));
        else out[c] = vfma(n[i], V[j], vfma(V[i], n[j], S.cX * X[c]));
    }
}

// ---- right-hand sides of Eq. StiffCons (Jaumann derivative) and Eq. BE -----------------------
// y = (sigma (6), dP = P - P_ref (3)) at the cell, reduced from each component's stencil as it is
// loaded: the value, the advection u.grad (central differences) and the 7-point Laplacian
template <class T>
struct Y9 {
    T c[9], adv[9], lap[9];
};

template <class T>
__device__ __forceinline__ void load_y9(const float* base, long long NP, const Nb<T>& q, const T* uc, Y9<T>& y)
{
    const T hu[3] = {0.5f * uc[0], 0.5f * uc[1], 0.5f * uc[2]};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        T dx, dy, dz, sum;
        fold(base + k * NP, q, y.c[k], dx, dy, dz, sum);
        y.adv[k] = vfma(hu[0], dx, vfma(hu[1], dy, hu[2] * dz));
        y.lap[k] = vfma(-6.f, y.c[k], sum);
    }
}

// u at the cell, Psi (xx, yy, zz, yz, xz, xy) and Om (01, 02, 12) of its gradient G_ij = d_i u_j
// (central differences)
template <class T>
struct Flow {
    T u[3], psi[6], om[3];
};

template <class T>
__device__ __forceinline__ void flow(const Args3& a, const Nb<T>& q, Flow<T>& f)
{
    T G[3][3], sum;              // 2 G
#pragma unroll
    for (int j = 0; j < 3; ++j) fold(a.u + j * a.NP, q, f.u[j], G[0][j], G[1][j], G[2][j], sum);
#pragma unroll
    for (int i = 0; i < 3; ++i) f.psi[i] = 0.5f * G[i][i];
    f.psi[3] = 0.25f * (G[1][2] + G[2][1]);
    f.psi[4] = 0.25f * (G[0][2] + G[2][0]);
    f.psi[5] = 0.25f * (G[0][1] + G[1][0]);
    f.om[0] = 0.25f * (G[0][1] - G[1][0]);
    f.om[1] = 0.25f * (G[0][2] - G[2][0]);
    f.om[2] = 0.25f * (G[1][2] - G[2][1]);
}

// the right-hand side at y, h the molecular field of its P (Eq. Ffunctional)
template <class T>
__device__ __forceinline__ void rhs9(const Args3& a, const Y9<T>& y, const Flow<T>& f, T* r)
{
    const T *s = y.c, *psi = f.psi;
    const T oa = f.om[0], ob = f.om[1], oc = f.om[2];
    const T P[3] = {y.c[6] + a.prx, y.c[7] + a.pry, y.c[8] + a.prz};
    Stiff<T> S;
    stiffness(a, P, S);
    // C Psi - C sigma / eta_p = C (Psi - sigma / eta_p): one contraction (C is linear in X)
    T X6[6], CX[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) X6[c] = vfma(-a.inv_eta, s[c], psi[c]);
    apply_c(S, X6, CX);
    // -(Omega s - s Omega) with Omega = (0 a b; -a 0 c; -b -c 0)
    T nJ[6];
    nJ[0] = -2.f * vfma(oa, s[5], ob * s[4]);
    nJ[1] = 2.f * vfma(oa, s[5], -1.f * (oc * s[3]));
    nJ[2] = 2.f * vfma(ob, s[4], oc * s[3]);
    nJ[3] = vfma(oa, s[4], vfma(ob, s[5], oc * (s[1] - s[2])));
    nJ[4] = vfma(ob, s[0] - s[2], vfma(oc, s[5], -1.f * (oa * s[3])));
    nJ[5] = vfma(oa, s[0] - s[1], -1.f * vfma(ob, s[3], oc * s[4]));
#pragma unroll
    for (int c = 0; c < 6; ++c) r[c] = vfma(a.Dp, y.lap[c], (CX[c] + nJ[c]) - y.adv[c]);
    // Eq. BE with h = (alpha + beta |P|^2) P - kappa lap P
    const T A = bulk(a, y.c[6], y.c[7], y.c[8]);
    const T rot[3] = {vfma(oa, P[1], ob * P[2]), vfma(oc, P[2], -1.f * (oa * P[0])), -1.f * vfma(ob, P[0], oc * P[1])};
    const T str[3] = {vfma(psi[0], P[0], vfma(psi[5], P[1], psi[4] * P[2])),
                      vfma(psi[5], P[0], vfma(psi[1], P[1], psi[3] * P[2])),
                      vfma(psi[4], P[0], vfma(psi[3], P[1], psi[2] * P[2]))};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const T h = vfma(A, P[i], (-a.kappa) * y.lap[6 + i]);
        r[6 + i] = vfma(-a.Gamma, h, vfma(a.xi, str[i], -1.f * (rot[i] + y.adv[6 + i])));
    }
}

// n planes of a row of 32 cells, a.ahead cells further on, into L2 (one lane per row)
__device__ __forceinline__ void prefetch_rows(const Args3& a, const float* base, int n, int c)
{
    if (c + a.ahead >= a.NP) return;
    const float* p = base + c + a.ahead;
    for (int k = 0; k < n; ++k, p += a.NP) asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// ---- kernels ---------------------------------------------------------------------------------

// row: the row i of sigma^E_ij wanted (-1: all)
__global__ void __launch_bounds__(NT) k3_molecular(const __grid_constant__ Args3 a, const float* dP, int row)
{
    pdl_wait();
    pdl_trigger();
    Cell q;
    if (!cell_of(a, q)) return;
    float v[3][7];                  // stencils of dP = P - P_ref
#pragma unroll
    for (int i = 0; i < 3; ++i) stencil(dP + i * a.NP, q, v[i]);
    const float A = bulk(a, v[0][0], v[1][0], v[2][0]);
    const float P[3] = {a.prx + v[0][0], a.pry + v[1][0], a.prz + v[2][0]};
    float h[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) h[i] = A * P[i] - a.kappa * lap7(v[i]);
    float gP[3][3];                 // gP[i][k] = d_i P_k
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) gP[i][k] = dif(v[k], i);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (row >= 0 && i != row) continue;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float Pi = P[i], Pj = P[j];
            const float gg = gP[i][0] * gP[j][0] + gP[i][1] * gP[j][1] + gP[i][2] * gP[j][2];
            a.sE[(i * 3 + j) * a.NP + q.c] = -0.5f * (Pi * h[j] - h[i] * Pj) + 0.5f * a.xi * (Pi * h[j] + h[i] * Pj)
                                             - a.kappa * gg;
        }
    }
}

// Fixed-order sums of the readout values v[7] of a CTA into out[7]: FP32 within each warp (a
// warp's cells are 32 consecutive FP32 values), FP64 across the warps, one thread per value (FP64
// is a narrow unit on this GPU: seven short chains, not one long one).
__device__ __forceinline__ void cta_sum7(const float* v, double* out, float* sm)
{
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        float x = v[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) sm[wid * 7 + k] = x;
    }
    __syncthreads();
    if (tid < 7) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) s += (double)sm[w * 7 + tid];
        out[tid] = s;
    }
}

// fixed-order FP64 block sum of v[7] (thread 0 returns the totals)
__device__ __forceinline__ void block_sum7(double* v, double* sm)
{
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        double x = v[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) sm[wid * 7 + k] = x;
    }
    __syncthreads();
    if (tid == 0) {
        for (int k = 0; k < 7; ++k) {
            double s = 0.0;
            for (int w = 0; w < NT / 32; ++w) s += sm[w * 7 + k];
            v[k] = s;
        }
    }
}

// the step's collision and streaming; MINB: CTAs per SM that the registers leave room for
template <int MINB>
__global__ void __launch_bounds__(NT, MINB) k3_collide(const __grid_constant__ Args3 a)
{
    pdl_wait();
    pdl_trigger();
    __shared__ float sRedF[(NT / 32) * 7];
    Cell q;
    const bool in = cell_of(a, q);
    float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (in) {
        // F_i = d_j sigma^p_ij + d_j sigma^E_ij + f_ext,i; every load ahead of the sums
        float F[3] = {a.fx, a.fy, a.fz};
        const int nb[3][2] = {{q.xp, q.xm}, {q.yp, q.ym}, {q.zp, q.zm}};
        float dp[9], de[9], d[NQ];
#pragma unroll
        for (int n = 0; n < NQ; ++n) d[n] = a.src[(long long)n * a.NP + q.c];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const float* sp = a.src + (long long)(PL_S + sym6(k / 3, k % 3)) * a.NP;
            dp[k] = sp[nb[k % 3][0]] - sp[nb[k % 3][1]];
        }
        if (a.ericksen) {
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const float* se = a.sE + (long long)k * a.NP;
                de[k] = se[nb[k % 3][0]] - se[nb[k % 3][1]];
            }
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            F[k / 3] += 0.5f * dp[k];
            if (a.ericksen) F[k / 3] += 0.5f * de[k];
        }
        float drho = 0.f, jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
        for (int n = 0; n < NQ; ++n) {
            drho += d[n];
            jx += (float)CX[n] * d[n];
            jy += (float)CY[n] * d[n];
            jz += (float)CZ[n] * d[n];
        }
        const float rho = a.rho0 + drho;
        const float ir = 1.f / rho;
        const float ux = (jx + 0.5f * F[0]) * ir, uy = (jy + 0.5f * F[1]) * ir, uz = (jz + 0.5f * F[2]) * ir;
        a.u[q.c] = ux;
        a.u[a.NP + q.c] = uy;
        a.u[2 * a.NP + q.c] = uz;
        // BGK with the Guo source: d* = d - (d - d_eq)/tau + (1 - 1/(2 tau)) w [3 (c - u) + 9 (c.u) c].F,
        // d_eq = w (drho + rho (3 c.u + 9/2 (c.u)^2 - 3/2 u.u)); pushed to x + c_n (periodic: the
        // neighbour offsets of the cell, combined per direction)
        const float rq = 1.5f * rho * (ux * ux + uy * uy + uz * uz);
        const float uF3 = 3.f * (ux * F[0] + uy * F[1] + uz * F[2]);
        const int ox[2] = {q.xp - q.c, q.xm - q.c}, oy[2] = {q.yp - q.c, q.ym - q.c}, oz[2] = {q.zp - q.c, q.zm - q.c};
        const float keep = 1.f - a.tau_inv;
        auto push = [&](int n, float out) {
            int dstc = q.c;
            if (CX[n]) dstc += ox[CX[n] > 0 ? 0 : 1];
            if (CY[n]) dstc += oy[CY[n] > 0 ? 0 : 1];
            if (CZ[n]) dstc += oz[CZ[n] > 0 ? 0 : 1];
            a.dst[(long long)n * a.NP + dstc] = out;
        };
        // rest population, then each direction n with its opposite n + 1 (the order of
        // include/lb3d.h pairs them) from the even and odd parts in c of d_eq and of the source
        const float base = drho - rq;
        push(0, keep * d[0] + a.tau_inv * (wq(0) * base) + (a.guo * wq(0)) * (-uF3));
#pragma unroll
        for (int n = 1; n < NQ; n += 2) {
            float cu = 0.f, cF = 0.f;
            if (CX[n]) { cu += CX[n] > 0 ? ux : -ux; cF += CX[n] > 0 ? F[0] : -F[0]; }
            if (CY[n]) { cu += CY[n] > 0 ? uy : -uy; cF += CY[n] > 0 ? F[1] : -F[1]; }
            if (CZ[n]) { cu += CZ[n] > 0 ? uz : -uz; cF += CZ[n] > 0 ? F[2] : -F[2]; }
            const float w = wq(n), gw = a.guo * w;
            const float ev = a.tau_inv * (w * (base + 4.5f * rho * cu * cu));     // even part of d_eq / tau
            const float od = a.tau_inv * (w * (3.f * rho * cu));                   // odd part
            const float Sev = gw * (9.f * cu * cF - uF3), Sod = gw * (3.f * cF);
            push(n, keep * d[n] + (ev + od) + (Sev + Sod));
            push(n + 1, keep * d[n + 1] + (ev - od) + (Sev - Sod));
        }
        if (a.readout) {
            acc[0] = drho;
            acc[1] = jx; acc[2] = jy; acc[3] = jz;
            acc[4] = F[0]; acc[5] = F[1]; acc[6] = F[2];
        }
    }
    if (!a.readout) return;
    // readout: the CTA's sums; the groups of NT CTAs are added by the next kernel and the groups by
    // the one after (kernel boundaries order the writes: no fence or atomic in this kernel)
    const unsigned cta = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    cta_sum7(acc, a.partials + (long long)cta * 7, sRedF);
}

// One moment of the current state into out: rho - rho0 (axis -1: the populations alone), or a component of
// u (its component of the force, from sigma^p and the row of sigma^E that k3_molecular has written).
// A readout asks for one field: forming all four moments each time read 34 planes of stress for one.
__global__ void __launch_bounds__(NT) k3_moment(const __grid_constant__ Args3 a, int axis, float* out)
{
    Cell q;
    if (!cell_of(a, q)) return;
    float drho = 0.f, jn = 0.f;
#pragma unroll
    for (int n = 0; n < NQ; ++n) {
        const float d = a.src[(long long)n * a.NP + q.c];
        drho += d;
        const int c = axis == 0 ? CX[n] : (axis == 1 ? CY[n] : CZ[n]);
        jn += (float)c * d;
    }
    if (axis < 0) {
        out[q.c] = drho;
        return;
    }
    float F = axis == 0 ? a.fx : (axis == 1 ? a.fy : a.fz);
    const int nb[3][2] = {{q.xp, q.xm}, {q.yp, q.ym}, {q.zp, q.zm}};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float* sp = a.src + (long long)(PL_S + sym6(axis, j)) * a.NP;
        F += 0.5f * (sp[nb[j][0]] - sp[nb[j][1]]);
        if (a.ericksen) {
            const float* se = a.sE + (long long)(axis * 3 + j) * a.NP;
            F += 0.5f * (se[nb[j][0]] - se[nb[j][1]]);
        }
    }
    out[q.c] = (jn + 0.5f * F) * (1.f / (a.rho0 + drho));
}

// Readout, second level (in k3_predict): CTA g < groups adds the sums of CTAs g NT .. g NT + NT - 1
// of k3_collide in a fixed tree.
__device__ __forceinline__ void readout_groups(const Args3& a, double* sm)
{
    const unsigned n_ctas = a.n_ctas;
    const unsigned cta = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    const unsigned n_grp = (n_ctas + NT - 1) / NT;
    if (!a.readout || cta >= n_grp) return;
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const unsigned g0 = cta * NT;
    double s[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (g0 + tid < n_ctas) {
#pragma unroll
        for (int k = 0; k < 7; ++k) s[k] = a.partials[(long long)(g0 + tid) * 7 + k];
    }
    block_sum7(s, sm);
    if (tid == 0)
        for (int k = 0; k < 7; ++k) a.gpartials[(long long)cta * 7 + k] = s[k];
}

// Readout, last level (in k3_correct, CTA 0): the group sums, each thread a fixed contiguous range,
// then the fixed tree; the row (t, mass, momentum, force) of the step.
__device__ __forceinline__ void readout_total(const Args3& a, double* sm)
{
    if (!a.readout || blockIdx.x + blockIdx.y + blockIdx.z != 0) return;
    const unsigned n_ctas = a.n_ctas;
    const unsigned n_grp = (n_ctas + NT - 1) / NT;
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const unsigned per = (n_grp + NT - 1) / NT;
    const unsigned b0 = min(n_grp, tid * per), b1 = min(n_grp, b0 + per);
    double s[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (unsigned b = b0; b < b1; ++b) {
#pragma unroll
        for (int k = 0; k < 7; ++k) s[k] += a.gpartials[(long long)b * 7 + k];
    }
    block_sum7(s, sm);
    if (tid == 0) {
        a.row[0] = (double)a.t;
        for (int k = 0; k < 7; ++k) {
            a.row[1 + k] = s[k];
            if (!isfinite(s[k])) atomicExch(a.err_nonfinite, 1);
        }
    }
}

// Predictor and corrector: streaming stencil kernels bound by instruction issue and load latency (63
// stencil points of y, 21 of u), so they take two cells per thread where nx is even: half the loads and
// arithmetic per cell, 16 warps of two cells per SM against 24 of one.
template <class T, int MINB>
__global__ void __launch_bounds__(NT, MINB) k3_predict(const __grid_constant__ Args3 a)
{
    pdl_wait();
    pdl_trigger();
    __shared__ double sRed[(NT / 32) * 7];
    readout_groups(a, sRed);
    Nb<T> q;
    if (!nb_of(a, q)) return;
    if (a.ahead && threadIdx.x == 0) {
        prefetch_rows(a, a.u, 3, q.c);
        prefetch_rows(a, a.src + (long long)PL_S * a.NP, 9, q.c);
    }
    Flow<T> f;
    flow(a, q, f);
    Y9<T> y;
    load_y9(a.src + (long long)PL_S * a.NP, a.NP, q, f.u, y);
    T r[9];
    rhs9(a, y, f, r);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        stv(a.r0 + k * a.NP + q.c, r[k]);
        stv(a.ys + k * a.NP + q.c, y.c[k] + r[k]);
    }
}

template <class T, int MINB>
__global__ void __launch_bounds__(NT, MINB) k3_correct(const __grid_constant__ Args3 a)
{
    pdl_wait();
    pdl_trigger();
    __shared__ double sRed[(NT / 32) * 7];
    readout_total(a, sRed);
    Nb<T> q;
    if (!nb_of(a, q)) return;
    if (a.ahead && threadIdx.x == 0) {
        prefetch_rows(a, a.u, 3, q.c);
        prefetch_rows(a, a.ys, 9, q.c);
        prefetch_rows(a, a.src + (long long)PL_S * a.NP, 9, q.c);
        prefetch_rows(a, a.r0, 9, q.c);
    }
    Flow<T> f;
    flow(a, q, f);
    Y9<T> y;
    load_y9(a.ys, a.NP, q, f.u, y);
    T r[9];
    rhs9(a, y, f, r);
    // all loads ahead of the stores, which they may not be moved across
    T y0[9], r0[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        y0[k] = ldv<T>(a.src + (long long)(PL_S + k) * a.NP + q.c);
        r0[k] = ldv<T>(a.r0 + k * a.NP + q.c);
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) stv(a.dst + (long long)(PL_S + k) * a.NP + q.c, vfma(0.5f, r0[k] + r[k], y0[k]));
}

// out = plane + c (the readout of P = P_ref + dP)
__global__ void k3_add(const float* plane, float c, float* out, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = plane[i] + c;
}

// ---- host: the orientation-moment table (FP64) ------------------------------------------------

double langevin(double k)
{
    if (k < 0.05) {
        const double k2 = k * k;
        return k * (1.0 / 3.0 - k2 * (1.0 / 45.0 - k2 * (2.0 / 945.0 - k2 / 4725.0)));
    }
    return 1.0 / std::tanh(k) - 1.0 / k;
}

// concentration of the Fisher density with mean projection P (bisection on the increasing L)
double concentration(double P)
{
    if (P <= 0.0) return 0.0;
    double lo = 0.0, hi = 1.0;
    while (langevin(hi) < P) hi *= 2.0;
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (langevin(mid) < P) lo = mid;
        else hi = mid;
        if (hi - lo <= 1e-15 * hi) break;
    }
    return 0.5 * (lo + hi);
}

// <mu^2>, <mu^4> of exp(k mu) on [-1, 1]: the power series of both integrals below k = 4, the
// integration-by-parts recursion m_n = [1 or coth k] - (n / k) m_{n-1} above
void fisher_moments(double k, double& m2, double& m4)
{
    if (k < 4.0) {
        double s[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
        double t = 1.0;                  // k^j / j!
        for (int j = 0; j < 80; ++j) {
            for (int n = 0; n <= 4; n += 2)
                if ((n + j) % 2 == 0) s[n] += t * 2.0 / (n + j + 1);
            t *= k / (j + 1);
        }
        m2 = s[2] / s[0];
        m4 = s[4] / s[0];
        return;
    }
    const double c = 1.0 / std::tanh(k);
    const double m1 = c - 1.0 / k;
    m2 = 1.0 - 2.0 / k * m1;
    const double m3 = c - 3.0 / k * m2;
    m4 = 1.0 - 4.0 / k * m3;
}

void moment_table(double P_cap, std::vector<float>& out)
{
    out.resize(2 * (LUT_N + 1));
    for (int i = 0; i <= LUT_N; ++i) {
        const double P = P_cap * i / LUT_N;
        double m2, m4;
        fisher_moments(concentration(P), m2, m4);
        out[2 * i] = (float)m2;
        out[2 * i + 1] = (float)m4;
    }
}

// The coefficients of C:X per table entry (8 floats: cpp_n, g, cd_t, cs, cX, 0, 0, 0), in FP64:
// K(n) in the transversely isotropic basis about n (K2323 = (K2222 - K2233) / 2), the moment
// tensors M2 = A d + B pp, M4 = e1 pppp + e2 Sym(pp d) + e3 Sym(d d) of the Fisher density.
void coefficient_table(const lb3d_params& p, std::vector<float>& out)
{
    const double a5 = 0.5 * (p.K2222 - p.K2233), a3 = p.K2233, a4 = p.K1212 - a5, a2 = p.K1122 - a3;
    const double a1 = p.K1111 - 2.0 * a2 - a3 - 4.0 * a4 - 2.0 * a5;
    out.assign(8 * (LUT_N + 1), 0.f);
    for (int i = 0; i <= LUT_N; ++i) {
        double m2, m4;
        fisher_moments(concentration(p.P_cap * i / LUT_N), m2, m4);
        const double A = 0.5 * (1.0 - m2), B = 0.5 * (3.0 * m2 - 1.0);
        const double e3 = (A - B + m4) / 8.0, e2 = A - 5.0 * e3, e1 = B - 7.0 * e2;
        float* o = out.data() + 8 * i;
        o[0] = (float)(a1 * e1);
        o[1] = (float)(a1 * e2 + a2 * B);
        o[2] = (float)(a1 * e3 + 2.0 * a2 * A + a3);
        o[3] = (float)(2.0 * (a1 * e2 + a4 * B));
        o[4] = (float)(2.0 * (a1 * e3 + 2.0 * a4 * A + a5));
    }
}

}  // namespace v3

// ---- host: the handle --------------------------------------------------------------------------

struct lb3d_handle {
    lb3d_params p;
    cudaStream_t stream = nullptr;
    int n_sm = 152;
    long long NP = 0;
    float* state[2] = {nullptr, nullptr};
    int cur = 0;
    float* sE = nullptr;
    float* u = nullptr;
    float* ys = nullptr;
    float* r0 = nullptr;
    float* scratch = nullptr;     // one plane: a formed field on its way to the host
    float4* lut = nullptr;
    double* partials = nullptr;
    double* gpartials = nullptr;
    double* series = nullptr;
    int* err = nullptr;
    long long t = 0;
    long long rows = 0;           // readout rows written since lb3d_init_fields
    bool ready = false;
    bool timing = false;
    std::vector<cudaEvent_t> ev;
    size_t ev_used = 0;
    std::string msg;
};

namespace {

int fail(lb3d_handle* h, int code, const char* fmt, ...)
{
    if (h) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof buf, fmt, ap);
        va_end(ap);
        h->msg = buf;
    }
    return code;
}

#define CK3(h, call)                                                                                   \
    do {                                                                                               \
        cudaError_t e_ = (call);                                                                       \
        if (e_ != cudaSuccess)                                                                         \
            return fail(h, e_ == cudaErrorMemoryAllocation ? LB_ENOMEM : LB_ECUDA, "%s: %s", #call,     \
                        cudaGetErrorString(e_));                                                       \
    } while (0)

template <class T>
void dfree(T*& p)
{
    if (p) cudaFree(p);
    p = nullptr;
}

dim3 grid_of(const lb3d_handle* h)
{
    return dim3((unsigned)((h->p.nx + v3::BX - 1) / v3::BX), (unsigned)((h->p.ny + v3::BY - 1) / v3::BY),
                (unsigned)((h->p.nz + v3::BZ - 1) / v3::BZ));
}

v3::Args3 args_of(lb3d_handle* h)
{
    const lb3d_params& p = h->p;
    v3::Args3 a = {};
    a.src = h->state[h->cur];
    a.dst = h->state[h->cur ^ 1];
    a.sE = h->sE; a.u = h->u; a.ys = h->ys; a.r0 = h->r0;
    a.lut = h->lut;
    a.NP = h->NP;
    a.nx = p.nx; a.ny = p.ny; a.nz = p.nz;
    a.tau_inv = (float)(1.0 / p.tau);
    a.guo = (float)(1.0 - 0.5 / p.tau);
    a.rho0 = (float)p.rho0;
    a.inv_eta = (float)(1.0 / p.eta_p);
    a.Dp = (float)p.Dp;
    a.alpha = (float)p.alpha; a.beta = (float)p.beta; a.xi = (float)p.xi;
    a.Gamma = (float)p.Gamma; a.kappa = (float)p.kappa;
    a.P_cap = (float)p.P_cap;
    a.lut_scale = (float)(v3::LUT_N / p.P_cap);
    a.fx = (float)p.fext[0]; a.fy = (float)p.fext[1]; a.fz = (float)p.fext[2];
    a.prx = (float)p.P_ref[0]; a.pry = (float)p.P_ref[1]; a.prz = (float)p.P_ref[2];
    a.A0 = (float)(p.alpha + p.beta * (p.P_ref[0] * p.P_ref[0] + p.P_ref[1] * p.P_ref[1] + p.P_ref[2] * p.P_ref[2]));
    a.ericksen = p.ericksen;
    a.partials = h->partials;
    a.gpartials = h->gpartials;
    const dim3 g = grid_of(h);
    a.n_ctas = g.x * g.y * g.z;
    // one plane ahead where the state does not stay in L2 (measured at 256^3: 1.825 ms per step without,
    // 1.739, 1.763, 1.826 and 2.012 ms with 1, 2, 3 and 4 planes)
    a.ahead = h->NP * v3::NPL * 4 > (64LL << 20) ? (long long)p.nx * p.ny : 0;
    a.err_nonfinite = h->err;
    a.t = h->t;
    return a;
}

// launch with or without programmatic stream serialization
template <class K, class... A>
int launch3(lb3d_handle* h, const char* what, K kern, dim3 g, dim3 b, bool pdl, const A&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g;
    cfg.blockDim = b;
    cfg.stream = h->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
    if (e != cudaSuccess) return fail(h, LB_ECUDA, "%s: %s", what, cudaGetErrorString(e));
    return LB_OK;
}

}  // namespace

extern "C" {

int lb3d_create(const lb3d_params* p, lb3d_handle** out)
{
    if (!p || !out) return LB_EINVAL;
    *out = nullptr;
    if (p->nx < 3 || p->ny < 3 || p->nz < 3 || (long long)p->nx * p->ny * p->nz >= (1LL << 31) ||
        p->readout_every < 1 || p->max_samples < 1 || !(p->tau > 0.5) || !(p->eta_p > 0.0) ||
        !(p->P_cap > 0.0 && p->P_cap < 1.0) || !(p->rho0 > 0.0) || p->Dp < 0.0 || p->Gamma < 0.0 ||
        p->kappa < 0.0)
        return LB_EINVAL;
    // Heun on the 7-point Laplacian (eigenvalues down to -12) and on the relaxation of P: the
    // explicit bounds 12 D_p <= 2, 12 Gamma kappa <= 2, 2 Gamma |alpha| <= 2
    if (12.0 * p->Dp > 2.0 || 12.0 * p->Gamma * p->kappa > 2.0 || p->Gamma * std::fabs(p->alpha) > 1.0)
        return LB_EUNSTABLE;
    lb3d_handle* h = new lb3d_handle();
    h->p = *p;
    h->NP = (long long)p->nx * p->ny * p->nz;
    auto bail = [&](int code) {
        lb3d_destroy(h);
        return code;
    };
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&h->n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking);
    const size_t pb = sizeof(float) * (size_t)h->NP;
    const dim3 g = grid_of(h);
    const size_t n_ctas = (size_t)g.x * g.y * g.z;
    for (int b = 0; b < 2 && e == cudaSuccess; ++b) e = cudaMalloc(&h->state[b], v3::NPL * pb);
    if (e == cudaSuccess && p->ericksen) e = cudaMalloc(&h->sE, 9 * pb);
    if (e == cudaSuccess) e = cudaMalloc(&h->u, 3 * pb);
    if (e == cudaSuccess) e = cudaMalloc(&h->ys, 9 * pb);
    if (e == cudaSuccess) e = cudaMalloc(&h->r0, 9 * pb);
    if (e == cudaSuccess) e = cudaMalloc(&h->scratch, pb);
    if (e == cudaSuccess) e = cudaMalloc(&h->lut, sizeof(float4) * 2 * (v3::LUT_N + 1));
    const size_t n_grp = (n_ctas + v3::NT - 1) / v3::NT;
    if (e == cudaSuccess) e = cudaMalloc(&h->partials, sizeof(double) * 7 * n_ctas);
    if (e == cudaSuccess) e = cudaMalloc(&h->gpartials, sizeof(double) * 7 * n_grp);
    if (e == cudaSuccess) e = cudaMalloc(&h->series, sizeof(double) * 8 * (size_t)p->max_samples);
    if (e == cudaSuccess) e = cudaMalloc(&h->err, sizeof(int));
    if (e != cudaSuccess) return bail(e == cudaErrorMemoryAllocation ? LB_ENOMEM : LB_ECUDA);
    std::vector<float> lut;
    v3::coefficient_table(*p, lut);
    e = cudaMemcpy(h->lut, lut.data(), sizeof(float) * lut.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(h->err, 0, sizeof(int));
    if (e != cudaSuccess) return bail(LB_ECUDA);
    *out = h;
    return LB_OK;
}

void lb3d_destroy(lb3d_handle* h)
{
    if (!h) return;
    if (h->stream) cudaStreamSynchronize(h->stream);
    dfree(h->state[0]); dfree(h->state[1]);
    dfree(h->sE); dfree(h->u); dfree(h->ys); dfree(h->r0); dfree(h->scratch);
    dfree(h->lut); dfree(h->partials); dfree(h->gpartials); dfree(h->series); dfree(h->err);
    for (auto e : h->ev) cudaEventDestroy(e);
    if (h->stream) cudaStreamDestroy(h->stream);
    delete h;
}

const char* lb3d_last_error(const lb3d_handle* h) { return h ? h->msg.c_str() : "null handle"; }

int lb3d_init_fields(lb3d_handle* h, const double* P_init)
{
    if (!h) return LB_EINVAL;
    const size_t N = (size_t)h->NP, pb = sizeof(float) * N;
    CK3(h, cudaStreamSynchronize(h->stream));
    // fluid at rest at rho0: every shifted population is 0; sigma^p = 0
    CK3(h, cudaMemset(h->state[0], 0, (size_t)v3::PL_P * pb));
    if (P_init) {
        std::vector<float> P(3 * N);
        for (int c = 0; c < 3; ++c)
            for (size_t i = 0; i < N; ++i) P[c * N + i] = (float)(P_init[c * N + i] - h->p.P_ref[c]);
        CK3(h, cudaMemcpy(h->state[0] + (size_t)v3::PL_P * N, P.data(), 3 * pb, cudaMemcpyHostToDevice));
    } else {
        // P = 0: dP = -P_ref
        std::vector<float> P(3 * N);
        for (int c = 0; c < 3; ++c)
            for (size_t i = 0; i < N; ++i) P[c * N + i] = (float)(-h->p.P_ref[c]);
        CK3(h, cudaMemcpy(h->state[0] + (size_t)v3::PL_P * N, P.data(), 3 * pb, cudaMemcpyHostToDevice));
    }
    CK3(h, cudaMemset(h->state[1], 0, v3::NPL * pb));
    CK3(h, cudaMemset(h->err, 0, sizeof(int)));
    h->cur = 0;
    h->t = 0;
    h->rows = 0;
    h->ready = true;
    return LB_OK;
}

int lb3d_step(lb3d_handle* h, int64_t n)
{
    if (!h) return LB_EINVAL;
    if (n < 0) return fail(h, LB_EINVAL, "n < 0");
    if (!h->ready) return fail(h, LB_ESTATE, "lb3d_init_fields not called");
    const dim3 g = grid_of(h), b(v3::BX, v3::BY, v3::BZ);
    // Few CTAs (at most two per SM): the kernels are bound by the latency of their loads, and registers for
    // more of them in flight pay (us per step, 16x12x8: 11.0 -> 10.3; 32^3: 13.3 -> 11.5; 44x38x30: 17.9 ->
    // 15.2, where two cells per thread take 18.8; beyond, 64^3 32.0 -> 34.0, 128^3 236 -> 262).  Else two
    // cells per thread where rows of pairs start at even indices (128^3 236 -> 228, 256^3 1.92 -> 1.74 ms),
    // CTAs of 32 x 8 x 2 cells.
    const bool few = (long long)g.x * g.y * g.z <= 2LL * h->n_sm;
    const bool pairs = !few && h->p.nx % 2 == 0;
    const dim3 b2(16, 8, 2), g2((unsigned)((h->p.nx / 2 + 15) / 16), (unsigned)((h->p.ny + 7) / 8), (unsigned)((h->p.nz + 1) / 2));
    for (int64_t k = 0; k < n; ++k) {
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        if (h->timing) {
            for (int i = 0; i < 2; ++i) {
                if (h->ev_used == h->ev.size()) {
                    cudaEvent_t e;
                    CK3(h, cudaEventCreate(&e));
                    h->ev.push_back(e);
                }
                (i ? e1 : e0) = h->ev[h->ev_used++];
            }
            CK3(h, cudaEventRecord(e0, h->stream));
        }
        v3::Args3 a = args_of(h);
        a.readout = (h->t % h->p.readout_every) == 0;
        if (a.readout) {
            a.row = h->series + (size_t)(h->rows % h->p.max_samples) * 8;
            h->rows += 1;
        }
        const bool pdl = !h->timing;
        int rc = LB_OK;
        if (h->p.ericksen)
            rc = launch3(h, "k3_molecular", v3::k3_molecular, g, b, pdl, a, a.src + (long long)v3::PL_P * h->NP, -1);
        if (!rc) rc = (few ? launch3(h, "k3_collide", v3::k3_collide<2>, g, b, pdl, a) : launch3(h, "k3_collide", v3::k3_collide<4>, g, b, pdl, a));
        if (!rc)
            rc = pairs ? launch3(h, "k3_predict", v3::k3_predict<float2, 2>, g2, b2, pdl, a)
                 : few ? launch3(h, "k3_predict", v3::k3_predict<float, 2>, g, b, pdl, a)
                       : launch3(h, "k3_predict", v3::k3_predict<float, 3>, g, b, pdl, a);
        if (!rc)
            rc = pairs ? launch3(h, "k3_correct", v3::k3_correct<float2, 2>, g2, b2, pdl, a)
                 : few ? launch3(h, "k3_correct", v3::k3_correct<float, 2>, g, b, pdl, a)
                       : launch3(h, "k3_correct", v3::k3_correct<float, 3>, g, b, pdl, a);
        if (rc) return rc;
        if (h->timing) CK3(h, cudaEventRecord(e1, h->stream));
        h->cur ^= 1;
        h->t += 1;
    }
    return LB_OK;
}

int lb3d_sync(lb3d_handle* h)
{
    if (!h) return LB_EINVAL;
    CK3(h, cudaStreamSynchronize(h->stream));
    int err = 0;
    CK3(h, cudaMemcpy(&err, h->err, sizeof(int), cudaMemcpyDeviceToHost));
    if (err) {
        CK3(h, cudaMemset(h->err, 0, sizeof(int)));
        return fail(h, LB_ENONFINITE, "a readout sum became NaN/Inf");
    }
    return LB_OK;
}

int64_t lb3d_time(const lb3d_handle* h) { return h ? h->t : -1; }

int lb3d_readout(lb3d_handle* h, int32_t field, float* dst, size_t count, int32_t dst_is_device)
{
    if (!h || !dst) return fail(h, LB_EINVAL, "null argument");
    if (field < 0 || field >= LB3D_N_FIELDS) return fail(h, LB_EINVAL, "unknown field %d", field);
    if (count < (size_t)h->NP) return fail(h, LB_EINVAL, "need %lld values", h->NP);
    if (!h->ready) return fail(h, LB_ESTATE, "lb3d_init_fields not called");
    // a formed field goes straight to memory of this device, or through the handle's scratch plane
    const float* srcp = nullptr;
    const bool direct = dst_is_device && vlb::device_floats(dst, sizeof(float) * (size_t)h->NP);
    float* out = direct ? dst : h->scratch;
    int rc = LB_OK;
    if (field <= 3) {
        v3::Args3 a = args_of(h);
        const dim3 g = grid_of(h), b(v3::BX, v3::BY, v3::BZ);
        if (h->p.ericksen && field > 0)
            rc = launch3(h, "k3_molecular", v3::k3_molecular, g, b, false, a, a.src + (long long)v3::PL_P * h->NP, field - 1);
        if (!rc) rc = launch3(h, "k3_moment", v3::k3_moment, g, b, false, a, field - 1, out);
    } else if (field < LB3D_FIELD_P) {
        srcp = h->state[h->cur] + (size_t)(v3::PL_S + field - LB3D_FIELD_SIGMA) * h->NP;
    } else if (field < LB3D_FIELD_POP0) {
        const int c = field - LB3D_FIELD_P;
        const float* plane = h->state[h->cur] + (size_t)(v3::PL_P + c) * h->NP;
        rc = launch3(h, "k3_add", v3::k3_add, dim3(1024), dim3(256), false, plane, (float)h->p.P_ref[c], out, h->NP);
    } else {
        srcp = h->state[h->cur] + (size_t)(field - LB3D_FIELD_POP0) * h->NP;
    }
    if (rc) return rc;
    if (!srcp && !direct) srcp = h->scratch;
    if (srcp)
        CK3(h, cudaMemcpyAsync(dst, srcp, sizeof(float) * (size_t)h->NP,
                               dst_is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, h->stream));
    CK3(h, cudaStreamSynchronize(h->stream));
    return LB_OK;
}

int lb3d_series(lb3d_handle* h, double* dst, int32_t max_rows, int32_t* rows_written)
{
    if (!h || !dst || max_rows < 0) return fail(h, LB_EINVAL, "bad argument");
    CK3(h, cudaStreamSynchronize(h->stream));
    const long long cap = h->p.max_samples;
    const long long n = std::min<long long>(h->rows, cap);
    const long long first = h->rows - n;
    std::vector<double> all((size_t)cap * 8);
    CK3(h, cudaMemcpy(all.data(), h->series, sizeof(double) * all.size(), cudaMemcpyDeviceToHost));
    const long long k = std::min<long long>(n, max_rows);
    for (long long i = 0; i < k; ++i) {
        const long long slot = (first + i) % cap;
        memcpy(dst + 8 * i, all.data() + 8 * slot, sizeof(double) * 8);
    }
    if (rows_written) *rows_written = (int32_t)k;
    return LB_OK;
}

int lb3d_timing(lb3d_handle* h, int32_t enable)
{
    if (!h) return LB_EINVAL;
    CK3(h, cudaStreamSynchronize(h->stream));
    h->timing = enable != 0;
    h->ev_used = 0;
    return LB_OK;
}

int lb3d_kernel_time(lb3d_handle* h, double* ms, int64_t* steps)
{
    if (!h) return LB_EINVAL;
    CK3(h, cudaStreamSynchronize(h->stream));
    double tot = 0.0;
    for (size_t i = 0; i + 1 < h->ev_used; i += 2) {
        float m = 0.f;
        CK3(h, cudaEventElapsedTime(&m, h->ev[i], h->ev[i + 1]));
        tot += m;
    }
    if (ms) *ms = tot;
    if (steps) *steps = (int64_t)(h->ev_used / 2);
    return LB_OK;
}

int32_t lb3d_launches_per_step(const lb3d_handle* h) { return h ? (h->p.ericksen ? 4 : 3) : 0; }

int32_t lb3d_moment_table(double P_cap, float* dst, int32_t max_entries)
{
    if (!(P_cap > 0.0 && P_cap < 1.0)) return LB_EINVAL;
    if (!dst) return v3::LUT_N + 1;
    if (max_entries < v3::LUT_N + 1) return LB_EINVAL;
    std::vector<float> t;
    v3::moment_table(P_cap, t);
    memcpy(dst, t.data(), sizeof(float) * t.size());
    return v3::LUT_N + 1;
}

double lb3d_bytes_per_cell(const lb3d_handle* h) { return h ? 2.0 * v3::NPL * sizeof(float) : 0.0; }

}  // extern "C"
