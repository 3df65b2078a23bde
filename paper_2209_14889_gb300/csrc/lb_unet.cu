// lb_unet.cu -- the network of the learned stepper: a 4-level convolutional U-Net on NHWC BF16
// activations with FP32 accumulation, forward and backward, trained on the GPU.
//
// Convolutions (3x3, stride 1, zero padding) are implicit GEMMs on the tensor cores (lb_conv.cu):
//   forward      y[p, o]  = b[o] + sum_{t, c} x[p + off_t, c] w[t, o, c]      (M = pixels, N = Co,
//                                                                           K = 9 Ci)
//   data grad    gx[q, c] = sum_{t', o} gz[q + off_t', o] w'[t', c, o],  w'[t'] = w[8 - t']^T
//                (the forward kernel on the flipped, transposed weights)
//   weight grad  gw[t, o, c] = sum_p gz[p, o] x[p + off_t, c]                (M = Ci, N = Co,
//                                                                           K = pixels)
// with off_t = (t / 3 - 1, t % 3 - 1), on tcgen05 (the forward and the data gradient on mma.sync by
// choice: lb_conv_kernel).  Weight gradients are reduced over pixel tiles in a fixed order (per-CTA
// partials, then a sum over CTAs), so training is bitwise reproducible.
// Joins: 2x2 average pooling, nearest 2x upsampling written into a channel slice of the
// concatenation buffer (the skip is written there by its producing convolution), LeakyReLU
// (slope 0.1).  The activation, the upsampled copy and, on the way back, the LeakyReLU gradient of
// the layer below are written by the convolution that produces the values; the gradients of the
// joins take the LeakyReLU gradient along.  Optimiser: Adam on FP32 master weights.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/lb.h"
#include "lb_conv.h"
#include "lb_device_ptr.h"
#include "lb_internal.h"

namespace vlb {
namespace net {

// ------------------------------------------------------------------ joins and pointwise
//
// Eight channels (16 bytes) per thread: memory-bound passes, and with one channel per thread they
// spent most of their time on the index divisions (2x upsampling of 64 channels to 4 x 256^2: 75 us
// for 42 MB).

struct Oct {
    float v[8];
};
__device__ __forceinline__ Oct ld8(const bf16* p)
{
    const uint4 q = *reinterpret_cast<const uint4*>(p);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&q);
    Oct o;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 f = __bfloat1622float2(h[e]);
        o.v[2 * e] = f.x;
        o.v[2 * e + 1] = f.y;
    }
    return o;
}
__device__ __forceinline__ void st8(bf16* p, const Oct& o)
{
    uint4 q;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&q);
#pragma unroll
    for (int e = 0; e < 4; ++e) h[e] = __floats2bfloat162_rn(o.v[2 * e], o.v[2 * e + 1]);
    *reinterpret_cast<uint4*>(p) = q;
}
__device__ __forceinline__ float rbf(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// pixel (b, y, x) and channel octet c of unit i of a [B][H][W][C8 octets] grid
struct Unit {
    int b, y, x, c;
    __device__ __forceinline__ Unit(unsigned i, int H, int W, int C8)
    {
        unsigned r = i / (unsigned)C8;
        c = (int)(i - r * (unsigned)C8) * 8;
        unsigned q = r / (unsigned)W;
        x = (int)(r - q * (unsigned)W);
        b = (int)(q / (unsigned)H);
        y = (int)(q - (unsigned)b * (unsigned)H);
    }
};

// gz = g * LeakyReLU'(from the sign of the activation output m), g a BF16 value
__device__ __forceinline__ void leaky_grad(Oct& g, const bf16* m)
{
    const Oct v = ld8(m);
#pragma unroll
    for (int e = 0; e < 8; ++e) g.v[e] = v.v[e] > 0.f ? g.v[e] : SLOPE * g.v[e];
}

// gz = g LeakyReLU'(y) (dense [P][C], C = 8 C8; the mma.sync convolution's own pass)
__global__ void k_leaky_bwd(const bf16* y, long long ldy, int yoff, bf16* g, long long P, int C8)
{
    pdl_wait();
    pdl_trigger();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P * C8) return;
    const long long p = i / C8;
    const int c = (int)(i - p * C8) * 8;
    Oct o = ld8(g + i * 8);
    leaky_grad(o, y + p * ldy + yoff + c);
    st8(g + i * 8, o);
}

// FP32 -> BF16 (dense, n a multiple of 8)
__global__ void k_to_bf16(const float* x, long long n, bf16* y)
{
    pdl_wait();
    pdl_trigger();
    const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * 8;
    if (i >= n) return;
    Oct o;
    if (((uintptr_t)x & 15) == 0) {
        const float4 a = *reinterpret_cast<const float4*>(x + i), b = *reinterpret_cast<const float4*>(x + i + 4);
        o = Oct{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
    } else {                                     // a caller's gradient at any address
        for (int e = 0; e < 8; ++e) o.v[e] = x[i + e];
    }
    st8(y + i, o);
}

// y[b, i, j, c] = mean of x[b, 2i + {0,1}, 2j + {0,1}, c]  (x: stride ldx, offset xoff; output H x W)
__global__ void k_pool2(const bf16* x, long long ldx, int xoff, unsigned n, int H, int W, int C8, bf16* y)
{
    pdl_wait();
    pdl_trigger();
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Unit u(i, H, W, C8);
    Oct s = {{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const Oct v = ld8(x + (((long long)u.b * 2 * H + 2 * u.y + (q >> 1)) * 2 * W + 2 * u.x + (q & 1)) * ldx + xoff + u.c);
#pragma unroll
        for (int e = 0; e < 8; ++e) s.v[e] += v.v[e];
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) s.v[e] *= 0.25f;
    st8(y + (long long)i * 8, s);
}

// g[b, y, x, c] = (gp[b, y/2, x/2, c] / 4 + gs[b, y, x, c]) LeakyReLU'(m[b, y, x, c])
// (gs: stride lds, offset soff; m: stride ldm, offset moff; output H x W)
__global__ void k_pool2_bwd_add(const bf16* gp, const bf16* gs, long long lds, int soff, const bf16* m, long long ldm,
                                int moff, unsigned n, int H, int W, int C8, bf16* g)
{
    pdl_wait();
    pdl_trigger();
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Unit u(i, H, W, C8);
    const long long p = ((long long)u.b * H + u.y) * W + u.x;
    const Oct a = ld8(gp + (((long long)u.b * (H / 2) + u.y / 2) * (W / 2) + u.x / 2) * (8 * C8) + u.c);
    Oct o = ld8(gs + p * lds + soff + u.c);
#pragma unroll
    for (int e = 0; e < 8; ++e) o.v[e] = rbf(0.25f * a.v[e] + o.v[e]);
    leaky_grad(o, m + p * ldm + moff + u.c);
    st8(g + (long long)i * 8, o);
}

// y[b, y, x, c] = x[b, y/2, x/2, c]   (y at full resolution H x W, stride ldy; the mma.sync form)
__global__ void k_up2(const bf16* x, unsigned n, int H, int W, int C8, bf16* y, long long ldy)
{
    pdl_wait();
    pdl_trigger();
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Unit u(i, H, W, C8);
    *reinterpret_cast<uint4*>(y + (((long long)u.b * H + u.y) * W + u.x) * ldy + u.c) =
        *reinterpret_cast<const uint4*>(x + (((long long)u.b * (H / 2) + u.y / 2) * (W / 2) + u.x / 2) * (8 * C8) + u.c);
}

// g[b, i, j, c] = (sum of gy[b, 2i + {0,1}, 2j + {0,1}, c]) LeakyReLU'(m[b, i, j, c])  (gy at 2H x 2W,
// stride ldg, offset 0; m dense; output H x W)
__global__ void k_up2_bwd(const bf16* gy, long long ldg, const bf16* m, unsigned n, int H, int W, int C8, bf16* g)
{
    pdl_wait();
    pdl_trigger();
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Unit u(i, H, W, C8);
    Oct s = {{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const Oct v = ld8(gy + (((long long)u.b * 2 * H + 2 * u.y + (q >> 1)) * 2 * W + 2 * u.x + (q & 1)) * ldg + u.c);
#pragma unroll
        for (int e = 0; e < 8; ++e) s.v[e] += v.v[e];
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) s.v[e] = rbf(s.v[e]);
    leaky_grad(s, m + (long long)i * 8);
    st8(g + (long long)i * 8, s);
}

// masked mean squared error: per-block partial sums of (pred - target)^2 and the gradient
// 2 (pred - target) mask / n
__global__ void k_mse(const float* pred, const float* target, const float* mask, long long P, float inv_n,
                      float* grad, double* part)
{
    __shared__ double red[256];
    double acc = 0.0;
    const long long n = P * 16;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float d = (pred[i] - target[i]) * mask[i & 15];
        acc += (double)d * d;
        grad[i] = 2.f * d * inv_n;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// Adam on FP32 master weights; writes the BF16 copy of the weights (not of the biases)
__global__ void k_adam(float* p, const float* g, float* m, float* v, long long n, float lr, float b1, float b2,
                       float eps, float c1, float c2, bf16* pb)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    p[i] = pi;
    if (pb) pb[i] = __float2bfloat16_rn(pi);
}

}  // namespace net
}  // namespace vlb

// ==================================================================== host side

using vlb::net::bf16;

namespace {

struct NetLayer {
    const char* name;
    int ci, co;
    bool act;
    long long w_off, b_off;      // offsets of w [9][co][ci] and b [co] in the flat parameter array
    long long p_off;             // offset of the layer in the packed weight arrays
};

// (name, Ci, Co, activation) in execution order; the same table as the FP64 oracle
const struct {
    const char* name;
    int ci, co;
    bool act;
} NET_LAYERS[] = {
    {"e0a", 16, 32, true},       {"e0b", 32, 32, true},  {"e1a", 32, 64, true},  {"e1b", 64, 64, true},
    {"e2a", 64, 96, true},       {"e2b", 96, 96, true},  {"bta", 96, 128, true}, {"btb", 128, 128, true},
    {"d2a", 128 + 96, 96, true}, {"d2b", 96, 96, true},  {"d1a", 96 + 64, 64, true}, {"d1b", 64, 64, true},
    {"d0a", 64 + 32, 32, true},  {"d0b", 32, 32, true},  {"head", 32, 16, false},
};
constexpr int N_LAYERS = 15;
enum { E0A, E0B, E1A, E1B, E2A, E2B, BTA, BTB, D2A, D2B, D1A, D1B, D0A, D0B, HEAD };

int blocks(long long n, int t = 256) { return (int)((n + t - 1) / t); }

}  // namespace

struct lb_net {
    int B = 0, H = 0, W = 0;
    cudaStream_t stream = nullptr;
    NetLayer L[N_LAYERS];
    long long n_params = 0;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    bf16* wb = nullptr;          // BF16 copy of the parameters (weights used)
    bf16 *wpf = nullptr, *wpd = nullptr;   // packed for the forward pass and for the data gradients
    bf16* wt = nullptr;          // flipped, transposed for the mma.sync data gradients
    // activations (BF16 NHWC)
    bf16 *x_in = nullptr, *t0 = nullptr, *cat0 = nullptr, *p1 = nullptr, *t1 = nullptr, *cat1 = nullptr;
    bf16 *p2 = nullptr, *t2 = nullptr, *cat2 = nullptr, *p3 = nullptr, *t3 = nullptr, *bt = nullptr;
    bf16 *u2 = nullptr, *d2 = nullptr, *u1 = nullptr, *d1 = nullptr, *u0 = nullptr, *d0 = nullptr;
    float* y = nullptr;          // head output FP32 [P0][16]
    float* gy = nullptr;         // loss gradient FP32 [P0][16]
    bf16* gs[6] = {};            // gradient scratch, P0 x 96 each
    float* part = nullptr;       // weight-gradient partials
    long long part_n = 0;
    double* lpart = nullptr;     // loss partials
    int adam_t = 0;
    std::vector<void*> allocs;
    std::string err;
};

namespace {

using namespace vlb::net;

int nfail(lb_net* n, int code, const std::string& msg)
{
    if (n) n->err = msg;
    return code;
}

#define NCK(n, call)                                                                   \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess) {                                                       \
            if (n) n->err = std::string(#call) + ": " + cudaGetErrorString(e_);        \
            return e_ == cudaErrorMemoryAllocation ? LB_ENOMEM : LB_ECUDA;             \
        }                                                                              \
    } while (0)

template <class T>
cudaError_t nalloc(lb_net* n, T** ptr, long long count)
{
    void* q = nullptr;
    cudaError_t e = cudaMalloc(&q, sizeof(T) * (size_t)count);
    if (e == cudaSuccess) {
        n->allocs.push_back(q);
        *ptr = static_cast<T*>(q);
    }
    return e;
}

// convolution kernel: 0 mma.sync, 1 tcgen05 (TMEM accumulators, the default)
int g_conv_kernel = 1;

unsigned units(long long n) { return (unsigned)((n + 255) / 256); }

// a convolution by the selected kernel; the mma.sync one has its extra outputs written by passes of
// their own
cudaError_t conv_run(const ConvArgs& a, cudaStream_t s, bool pdl)
{
    if (g_conv_kernel == 1) return conv_tc(a, s, pdl);
    cudaError_t e = conv_mma(a, s);
    const long long P = (long long)a.B * a.H * a.W;
    if (e == cudaSuccess && a.ym)
        e = launch_pdl(k_leaky_bwd, units(P * a.Co / 8), 256, 0, s, false, a.ym, a.ldm, a.moff, a.y, P, a.Co / 8);
    if (e == cudaSuccess && a.up)
        e = launch_pdl(k_up2, units(P * 4 * a.Co / 8), 256, 0, s, false, (const bf16*)a.y, (unsigned)(P * 4 * a.Co / 8),
                       2 * a.H, 2 * a.W, a.Co / 8, a.up, a.ldu);
    if (e == cudaSuccess && a.yf2)
        e = cudaMemcpyAsync(a.yf2, a.yf, sizeof(float) * P * a.ldy, cudaMemcpyDeviceToDevice, s);
    return e;
}

// the forms of the BF16 weights that the kernels read
cudaError_t refresh_weights(lb_net* n)
{
    static_assert(N_LAYERS <= PACK_MAX, "one launch packs every layer");
    PackArgs p = {};
    p.n = N_LAYERS;
    for (int l = 0; l < N_LAYERS; ++l) {
        const NetLayer& Ly = n->L[l];
        p.L[l] = PackLayer{n->wb + Ly.w_off, Ly.ci, Ly.co, n->wpf + Ly.p_off, n->wpd + Ly.p_off, n->wt + Ly.p_off};
    }
    return conv_pack(p, n->stream);
}

// forward of layer l: input (x, ldx, xoff) at resolution H x W -> output (y | yf, ldy, yoff), and
// optionally an upsampled copy (up, ldu) or a second FP32 copy (yf2)
cudaError_t layer_fwd(lb_net* n, int l, const bf16* x, long long ldx, int xoff, bf16* y, float* yf, long long ldy,
                      int yoff, int H, int W, bf16* up = nullptr, long long ldu = 0, float* yf2 = nullptr)
{
    const NetLayer& Ly = n->L[l];
    ConvArgs a = {};
    a.x = x; a.ldx = ldx; a.xoff = xoff;
    a.w = n->wb + Ly.w_off; a.wp = n->wpf + Ly.p_off; a.bias = n->p + Ly.b_off;
    a.y = y; a.yf = yf; a.ldy = ldy; a.yoff = yoff;
    a.B = n->B; a.H = H; a.W = W; a.Ci = Ly.ci; a.Co = Ly.co; a.act = Ly.act ? 1 : 0;
    a.up = up; a.ldu = ldu; a.yf2 = yf2;
    return conv_run(a, n->stream, l != E0A);
}

// backward of layer l given the gradient gz at its pre-activation output (dense [P][co]): weight and
// bias gradients, and into gx (dense [P][ci], if not null) the gradient at its input, taken through
// the LeakyReLU whose output is m (stride ldm, offset moff) if m is not null
cudaError_t layer_bwd(lb_net* n, int l, const bf16* x, long long ldx, int xoff, const bf16* gz, bf16* gx, const bf16* m,
                      long long ldm, int moff, int H, int W)
{
    const NetLayer& Ly = n->L[l];
    cudaError_t e = conv_wgrad(n->stream, x, ldx, xoff, gz, n->B, H, W, Ly.ci, Ly.co, n->part, n->part_n,
                               n->g + Ly.w_off, n->g + Ly.b_off, true);
    if (e != cudaSuccess || !gx) return e;
    ConvArgs a = {};
    a.x = gz; a.ldx = Ly.co;
    a.w = n->wt + Ly.p_off; a.wp = n->wpd + Ly.p_off;
    a.y = gx; a.ldy = Ly.ci;
    a.B = n->B; a.H = H; a.W = W; a.Ci = Ly.co; a.Co = Ly.ci;
    a.ym = m; a.ldm = ldm; a.moff = moff;
    return conv_run(a, n->stream, true);
}

// yout: a second copy of the output (device FP32 [P0][16]) or null
int net_forward(lb_net* n, float* yout)
{
    const int H = n->H, W = n->W, B = n->B;
    const int H1 = H / 2, W1 = W / 2, H2 = H / 4, W2 = W / 4, H3 = H / 8, W3 = W / 8;
    auto pool = [&](const bf16* x, long long ldx, int xoff, int h, int w, int C, bf16* y) {
        const unsigned u = (unsigned)((long long)B * h * w * C / 8);
        return launch_pdl(k_pool2, units(u), 256, 0, n->stream, true, x, ldx, xoff, u, h, w, C / 8, y);
    };
    NCK(n, layer_fwd(n, E0A, n->x_in, 16, 0, n->t0, nullptr, 32, 0, H, W));
    NCK(n, layer_fwd(n, E0B, n->t0, 32, 0, n->cat0, nullptr, 96, 64, H, W));
    NCK(n, pool(n->cat0, 96, 64, H1, W1, 32, n->p1));
    NCK(n, layer_fwd(n, E1A, n->p1, 32, 0, n->t1, nullptr, 64, 0, H1, W1));
    NCK(n, layer_fwd(n, E1B, n->t1, 64, 0, n->cat1, nullptr, 160, 96, H1, W1));
    NCK(n, pool(n->cat1, 160, 96, H2, W2, 64, n->p2));
    NCK(n, layer_fwd(n, E2A, n->p2, 64, 0, n->t2, nullptr, 96, 0, H2, W2));
    NCK(n, layer_fwd(n, E2B, n->t2, 96, 0, n->cat2, nullptr, 224, 128, H2, W2));
    NCK(n, pool(n->cat2, 224, 128, H3, W3, 96, n->p3));
    NCK(n, layer_fwd(n, BTA, n->p3, 96, 0, n->t3, nullptr, 128, 0, H3, W3));
    NCK(n, layer_fwd(n, BTB, n->t3, 128, 0, n->bt, nullptr, 128, 0, H3, W3, n->cat2, 224));
    NCK(n, layer_fwd(n, D2A, n->cat2, 224, 0, n->u2, nullptr, 96, 0, H2, W2));
    NCK(n, layer_fwd(n, D2B, n->u2, 96, 0, n->d2, nullptr, 96, 0, H2, W2, n->cat1, 160));
    NCK(n, layer_fwd(n, D1A, n->cat1, 160, 0, n->u1, nullptr, 64, 0, H1, W1));
    NCK(n, layer_fwd(n, D1B, n->u1, 64, 0, n->d1, nullptr, 64, 0, H1, W1, n->cat0, 96));
    NCK(n, layer_fwd(n, D0A, n->cat0, 96, 0, n->u0, nullptr, 32, 0, H, W));
    NCK(n, layer_fwd(n, D0B, n->u0, 32, 0, n->d0, nullptr, 32, 0, H, W));
    NCK(n, layer_fwd(n, HEAD, n->d0, 32, 0, nullptr, n->y, 16, 0, H, W, nullptr, 0, yout));
    NCK(n, cudaGetLastError());
    return LB_OK;
}

// gradients of sum(gy * y) for every parameter (overwritten), from the activations of the last
// forward; gy: FP32 [P0][16].  Every g below is taken through the LeakyReLU of the layer it enters.
int net_backward(lb_net* n, const float* gy)
{
    const int H = n->H, W = n->W, B = n->B;
    const int H1 = H / 2, W1 = W / 2, H2 = H / 4, W2 = W / 4, H3 = H / 8, W3 = W / 8;
    cudaStream_t s = n->stream;
    bf16 *A = n->gs[0], *Z = n->gs[1], *C = n->gs[2], *D = n->gs[3], *E = n->gs[4], *F = n->gs[5];
    const long long P0 = (long long)B * H * W;
    // gradient of the nearest upsampling (the first channels of a concatenation's gradient gy), at h x w
    auto up2_bwd = [&](const bf16* gy2, long long ldg, const bf16* m, int h, int w, int ch, bf16* g) {
        const unsigned u = (unsigned)((long long)B * h * w * ch / 8);
        return launch_pdl(k_up2_bwd, units(u), 256, 0, s, true, gy2, ldg, m, u, h, w, ch / 8, g);
    };
    // gradient of the pooling (gp) plus that of the skip (gs), at h x w
    auto pool_bwd = [&](const bf16* gp, const bf16* gs, long long lds, int soff, const bf16* m, int h, int w, int ch,
                        bf16* g) {
        const unsigned u = (unsigned)((long long)B * h * w * ch / 8);
        return launch_pdl(k_pool2_bwd_add, units(u), 256, 0, s, true, gp, gs, lds, soff, m, lds, soff, u, h, w, ch / 8, g);
    };
    NCK(n, launch_pdl(k_to_bf16, units(P0 * 2), 256, 0, s, false, gy, P0 * 16, Z));
    NCK(n, layer_bwd(n, HEAD, n->d0, 32, 0, Z, A, n->d0, 32, 0, H, W));               // A = g d0
    NCK(n, layer_bwd(n, D0B, n->u0, 32, 0, A, Z, n->u0, 32, 0, H, W));                // Z = g u0
    NCK(n, layer_bwd(n, D0A, n->cat0, 96, 0, Z, C, nullptr, 0, 0, H, W));             // C = g cat0
    NCK(n, up2_bwd(C, 96, n->d1, H1, W1, 64, A));                                     // A = g d1
    NCK(n, layer_bwd(n, D1B, n->u1, 64, 0, A, Z, n->u1, 64, 0, H1, W1));              // Z = g u1
    NCK(n, layer_bwd(n, D1A, n->cat1, 160, 0, Z, D, nullptr, 0, 0, H1, W1));          // D = g cat1
    NCK(n, up2_bwd(D, 160, n->d2, H2, W2, 96, A));                                    // A = g d2
    NCK(n, layer_bwd(n, D2B, n->u2, 96, 0, A, Z, n->u2, 96, 0, H2, W2));              // Z = g u2
    NCK(n, layer_bwd(n, D2A, n->cat2, 224, 0, Z, E, nullptr, 0, 0, H2, W2));          // E = g cat2
    NCK(n, up2_bwd(E, 224, n->bt, H3, W3, 128, A));                                   // A = g bt
    NCK(n, layer_bwd(n, BTB, n->t3, 128, 0, A, Z, n->t3, 128, 0, H3, W3));            // Z = g t3
    NCK(n, layer_bwd(n, BTA, n->p3, 96, 0, Z, F, nullptr, 0, 0, H3, W3));             // F = g p3
    NCK(n, pool_bwd(F, E, 224, 128, n->cat2, H2, W2, 96, A));                         // A = g e2
    NCK(n, layer_bwd(n, E2B, n->t2, 96, 0, A, Z, n->t2, 96, 0, H2, W2));              // Z = g t2
    NCK(n, layer_bwd(n, E2A, n->p2, 64, 0, Z, F, nullptr, 0, 0, H2, W2));             // F = g p2
    NCK(n, pool_bwd(F, D, 160, 96, n->cat1, H1, W1, 64, A));                          // A = g e1
    NCK(n, layer_bwd(n, E1B, n->t1, 64, 0, A, Z, n->t1, 64, 0, H1, W1));              // Z = g t1
    NCK(n, layer_bwd(n, E1A, n->p1, 32, 0, Z, F, nullptr, 0, 0, H1, W1));             // F = g p1
    NCK(n, pool_bwd(F, C, 96, 64, n->cat0, H, W, 32, A));                             // A = g e0
    NCK(n, layer_bwd(n, E0B, n->t0, 32, 0, A, Z, n->t0, 32, 0, H, W));                // Z = g t0
    NCK(n, layer_bwd(n, E0A, n->x_in, 16, 0, Z, nullptr, nullptr, 0, 0, H, W));
    return LB_OK;
}

}  // namespace

extern "C" {

int lb_net_create(int32_t batch, int32_t height, int32_t width, uint64_t seed, void* stream, lb_net** out)
{
    if (!out) return LB_EINVAL;
    *out = nullptr;
    if (batch < 1 || height < 8 || width < 8 || height % 8 || width % 8 || (long long)batch * height * width > (1LL << 28))
        return LB_EINVAL;
    lb_net* n = new lb_net();
    n->B = batch;
    n->H = height;
    n->W = width;
    n->stream = (cudaStream_t)stream;
    long long off = 0, poff = 0;
    for (int l = 0; l < N_LAYERS; ++l) {
        NetLayer& Ly = n->L[l];
        Ly.name = NET_LAYERS[l].name;
        Ly.ci = NET_LAYERS[l].ci;
        Ly.co = NET_LAYERS[l].co;
        Ly.act = NET_LAYERS[l].act;
        Ly.w_off = off;
        off += 9LL * Ly.ci * Ly.co;
        Ly.b_off = off;
        off += Ly.co;
        Ly.p_off = poff;
        poff += (conv_pack_elems(std::max(Ly.ci, Ly.co), std::max(Ly.ci, Ly.co)) + 7) / 8 * 8;
    }
    n->n_params = off;
    auto cleanup = [&](int code) { lb_net_destroy(n); return code; };
    const long long P0 = (long long)batch * height * width, P1 = P0 / 4, P2 = P0 / 16, P3 = P0 / 64;
    long long max_part = 0;
    for (int l = 0; l < N_LAYERS; ++l) max_part = std::max<long long>(max_part, 9LL * n->L[l].co * n->L[l].ci);
    max_part = std::max<long long>(max_part, 128) * 64;
    n->part_n = max_part;
    if (nalloc(n, &n->p, off) || nalloc(n, &n->g, off) || nalloc(n, &n->m, off) || nalloc(n, &n->v, off) ||
        nalloc(n, &n->wb, off) || nalloc(n, &n->wpf, poff) ||
        nalloc(n, &n->wpd, poff) || nalloc(n, &n->wt, poff) || nalloc(n, &n->x_in, P0 * 16) ||
        nalloc(n, &n->t0, P0 * 32) || nalloc(n, &n->cat0, P0 * 96) || nalloc(n, &n->p1, P1 * 32) ||
        nalloc(n, &n->t1, P1 * 64) || nalloc(n, &n->cat1, P1 * 160) || nalloc(n, &n->p2, P2 * 64) ||
        nalloc(n, &n->t2, P2 * 96) || nalloc(n, &n->cat2, P2 * 224) || nalloc(n, &n->p3, P3 * 96) ||
        nalloc(n, &n->t3, P3 * 128) || nalloc(n, &n->bt, P3 * 128) || nalloc(n, &n->u2, P2 * 96) ||
        nalloc(n, &n->d2, P2 * 96) || nalloc(n, &n->u1, P1 * 64) || nalloc(n, &n->d1, P1 * 64) ||
        nalloc(n, &n->u0, P0 * 32) || nalloc(n, &n->d0, P0 * 32) || nalloc(n, &n->y, P0 * 16) ||
        nalloc(n, &n->gy, P0 * 16) || nalloc(n, &n->part, max_part) || nalloc(n, &n->lpart, 1024))
        return cleanup(LB_ENOMEM);
    for (int i = 0; i < 6; ++i)
        if (nalloc(n, &n->gs[i], P0 * 96)) return cleanup(LB_ENOMEM);
    // He initialisation from a seeded generator (host, FP64 Box-Muller), zero biases
    std::vector<float> h(off, 0.f);
    uint64_t st = seed * 0x9E3779B97F4A7C15ULL + 1;
    auto next = [&]() {   // splitmix64
        uint64_t z = (st += 0x9E3779B97F4A7C15ULL);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        return z ^ (z >> 31);
    };
    for (int l = 0; l < N_LAYERS; ++l) {
        const NetLayer& Ly = n->L[l];
        const double sd = Ly.act ? std::sqrt(2.0 / (9.0 * Ly.ci)) : 0.1 * std::sqrt(1.0 / (9.0 * Ly.ci));
        for (long long i = 0; i < 9LL * Ly.ci * Ly.co; ++i) {
            const double u1 = ((next() >> 11) + 0.5) * (1.0 / 9007199254740992.0);
            const double u2 = ((next() >> 11) + 0.5) * (1.0 / 9007199254740992.0);
            h[Ly.w_off + i] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
        }
    }
    const int rc = lb_net_set_params(n, h.data(), off);
    if (rc != LB_OK) return cleanup(rc);
    if (cudaMemset(n->m, 0, sizeof(float) * off) != cudaSuccess || cudaMemset(n->v, 0, sizeof(float) * off) != cudaSuccess ||
        cudaMemset(n->g, 0, sizeof(float) * off) != cudaSuccess)
        return cleanup(LB_ECUDA);
    *out = n;
    return LB_OK;
}

int64_t lb_net_num_params(const lb_net* n) { return n ? n->n_params : -1; }

int lb_net_shape(const lb_net* n, int32_t* batch, int32_t* height, int32_t* width)
{
    if (!n || !batch || !height || !width) return LB_EINVAL;
    *batch = n->B;
    *height = n->H;
    *width = n->W;
    return LB_OK;
}

int lb_net_set_params(lb_net* n, const float* host, int64_t count)
{
    if (!n || !host) return LB_EINVAL;
    if (count != n->n_params) return nfail(n, LB_EINVAL, "parameter count mismatch");
    NCK(n, cudaMemcpyAsync(n->p, host, sizeof(float) * count, cudaMemcpyHostToDevice, n->stream));
    k_to_bf16<<<blocks(count / 8), 256, 0, n->stream>>>(n->p, count, n->wb);
    NCK(n, refresh_weights(n));
    NCK(n, cudaStreamSynchronize(n->stream));
    n->adam_t = 0;
    return LB_OK;
}

int lb_net_get_params(lb_net* n, float* host, int64_t count)
{
    if (!n || !host) return LB_EINVAL;
    if (count != n->n_params) return nfail(n, LB_EINVAL, "parameter count mismatch");
    NCK(n, cudaMemcpyAsync(host, n->p, sizeof(float) * count, cudaMemcpyDeviceToHost, n->stream));
    NCK(n, cudaStreamSynchronize(n->stream));
    return LB_OK;
}

int lb_net_get_grads(lb_net* n, float* host, int64_t count)
{
    if (!n || !host) return LB_EINVAL;
    if (count != n->n_params) return nfail(n, LB_EINVAL, "parameter count mismatch");
    NCK(n, cudaMemcpyAsync(host, n->g, sizeof(float) * count, cudaMemcpyDeviceToHost, n->stream));
    NCK(n, cudaStreamSynchronize(n->stream));
    return LB_OK;
}

int lb_net_forward(lb_net* n, const void* x, float* y)
{
    if (!n || !x) return LB_EINVAL;
    const long long P0 = (long long)n->B * n->H * n->W;
    NCK(n, cudaMemcpyAsync(n->x_in, x, sizeof(bf16) * P0 * 16, cudaMemcpyDeviceToDevice, n->stream));
    // the last convolution stores the output in y too, where a kernel may write; elsewhere a copy, which
    // handles or refuses the address
    const bool direct = y && vlb::device_floats(y, sizeof(float) * P0 * 16);
    const int rc = net_forward(n, direct ? y : nullptr);
    if (rc == LB_OK && y && !direct)
        NCK(n, cudaMemcpyAsync(y, n->y, sizeof(float) * P0 * 16, cudaMemcpyDeviceToDevice, n->stream));
    return rc;
}

const float* lb_net_output(const lb_net* n) { return n ? n->y : nullptr; }

int lb_net_backward(lb_net* n, const float* grad_out)
{
    if (!n || !grad_out) return LB_EINVAL;
    return net_backward(n, grad_out);
}

int lb_net_mse(lb_net* n, const float* target, const float* mask16, double* loss)
{
    if (!n || !target || !mask16) return LB_EINVAL;
    const long long P0 = (long long)n->B * n->H * n->W;
    float msum = 0.f;
    for (int c = 0; c < 16; ++c) msum += mask16[c];
    if (!(msum > 0.f)) return nfail(n, LB_EINVAL, "empty channel mask");
    float* mdev = reinterpret_cast<float*>(n->lpart + 512);   // 16 floats after the loss partials
    NCK(n, cudaMemcpyAsync(mdev, mask16, sizeof(float) * 16, cudaMemcpyHostToDevice, n->stream));
    const int nb = 256;
    k_mse<<<nb, 256, 0, n->stream>>>(n->y, target, mdev, P0, (float)(1.0 / ((double)P0 * msum)), n->gy, n->lpart);
    NCK(n, cudaGetLastError());
    if (loss) {
        std::vector<double> h(nb);
        NCK(n, cudaMemcpyAsync(h.data(), n->lpart, sizeof(double) * nb, cudaMemcpyDeviceToHost, n->stream));
        NCK(n, cudaStreamSynchronize(n->stream));
        double s = 0.0;
        for (int i = 0; i < nb; ++i) s += h[i];
        *loss = s / ((double)P0 * msum);
    }
    return LB_OK;
}

const float* lb_net_loss_grad(const lb_net* n) { return n ? n->gy : nullptr; }

int lb_net_adam(lb_net* n, float lr, float beta1, float beta2, float eps)
{
    if (!n || !(lr >= 0.f)) return LB_EINVAL;
    n->adam_t += 1;
    const float c1 = 1.f / (1.f - std::pow(beta1, (float)n->adam_t));
    const float c2 = 1.f / (1.f - std::pow(beta2, (float)n->adam_t));
    k_adam<<<blocks(n->n_params), 256, 0, n->stream>>>(n->p, n->g, n->m, n->v, n->n_params, lr, beta1, beta2, eps, c1,
                                                       c2, n->wb);
    NCK(n, cudaGetLastError());
    NCK(n, refresh_weights(n));
    return LB_OK;
}

int lb_net_train_step(lb_net* n, const void* x, const float* target, const float* mask16, float lr, double* loss)
{
    int rc = lb_net_forward(n, x, nullptr);
    if (rc == LB_OK) rc = lb_net_mse(n, target, mask16, loss);
    if (rc == LB_OK) rc = net_backward(n, n->gy);
    if (rc == LB_OK) rc = lb_net_adam(n, lr, 0.9f, 0.999f, 1e-8f);
    return rc;
}

int lb_net_activation(lb_net* n, int32_t which, void* host, int64_t bytes)
{
    if (!n || !host) return LB_EINVAL;
    const long long P0 = (long long)n->B * n->H * n->W, P1 = P0 / 4, P2 = P0 / 16, P3 = P0 / 64;
    const struct {
        const void* p;
        long long n;
    } T[] = {{n->x_in, P0 * 16}, {n->t0, P0 * 32}, {n->cat0, P0 * 96}, {n->p1, P1 * 32}, {n->t1, P1 * 64},
             {n->cat1, P1 * 160}, {n->p2, P2 * 64}, {n->t2, P2 * 96}, {n->cat2, P2 * 224}, {n->p3, P3 * 96},
             {n->t3, P3 * 128}, {n->bt, P3 * 128}, {n->u2, P2 * 96}, {n->d2, P2 * 96}, {n->u1, P1 * 64},
             {n->d1, P1 * 64}, {n->u0, P0 * 32}, {n->d0, P0 * 32}};
    if (which < 0 || which >= (int)(sizeof T / sizeof T[0])) return nfail(n, LB_EINVAL, "no such activation");
    if (bytes != (int64_t)(T[which].n * sizeof(bf16))) return nfail(n, LB_EINVAL, "bytes mismatch");
    NCK(n, cudaMemcpyAsync(host, T[which].p, (size_t)bytes, cudaMemcpyDeviceToHost, n->stream));
    NCK(n, cudaStreamSynchronize(n->stream));
    return LB_OK;
}

const char* lb_net_last_error(const lb_net* n) { return n ? n->err.c_str() : "null network"; }

void lb_net_destroy(lb_net* n)
{
    if (!n) return;
    if (n->stream) cudaStreamSynchronize(n->stream);
    for (void* q : n->allocs) cudaFree(q);
    delete n;
}

// ---- single-layer entry points (the building blocks, for tests against the oracle) ----

int lb_conv_kernel(int32_t kernel)
{
    if (kernel != 0 && kernel != 1) return LB_EINVAL;
    g_conv_kernel = kernel;
    return LB_OK;
}

int lb_conv_status(void)
{
    int* const flag = conv_err_flag();
    if (!flag) return LB_OK;
    int e = 0;
    if (cudaMemcpy(&e, flag, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return LB_ECUDA;
    if (e) {
        const int z = 0;
        cudaMemcpy(flag, &z, sizeof(int), cudaMemcpyHostToDevice);
        return LB_ETIMEOUT;
    }
    return LB_OK;
}

}  // extern "C"

namespace {

// Stream-ordered scratch of the single-layer calls, from a pool of its own per device that keeps at
// most 64 MB between calls (the default pool would hand its memory back, and map it again, at every
// synchronisation) until lb_conv_release.
constexpr int MAX_DEVICES = 64;
std::mutex g_pool_mu;
cudaMemPool_t g_pools[MAX_DEVICES] = {};

cudaError_t scratch(void** p, size_t bytes, cudaStream_t s)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaMallocAsync(p, bytes, s);
    cudaMemPool_t pool;
    {
        std::lock_guard<std::mutex> lock(g_pool_mu);
        if (!g_pools[dev]) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            e = cudaMemPoolCreate(&g_pools[dev], &props);
            if (e != cudaSuccess) return e;
            uint64_t keep = 64ull << 20;
            cudaMemPoolSetAttribute(g_pools[dev], cudaMemPoolAttrReleaseThreshold, &keep);
        }
        pool = g_pools[dev];
    }
    return cudaMallocFromPoolAsync(p, bytes, pool, s);
}

// The end of a gradient call: its scratch given back and its work done, so that the results may be used from
// anywhere and a fault of its kernels is its own return code.
cudaError_t finish(void* p, cudaError_t e, cudaStream_t s)
{
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    const cudaError_t f = cudaFreeAsync(p, s);
    return e != cudaSuccess ? e : f;
}

int conv_code(cudaError_t e) { return e == cudaSuccess ? LB_OK : (e == cudaErrorMemoryAllocation ? LB_ENOMEM : LB_ECUDA); }

}  // namespace

extern "C" {

int lb_conv3x3(const void* x, int64_t ldx, int32_t xoff, const void* w, const float* bias, void* y, float* yf,
               int64_t ldy, int32_t yoff, int32_t B, int32_t H, int32_t W, int32_t Ci, int32_t Co, int32_t act,
               void* stream)
{
    if (!x || !w || (!y && !yf) || B < 1 || H < 1 || W < 1 || Ci < 16 || Co < 16 || Ci % 16 || Co % 8 || ldx % 8 ||
        xoff % 8 || ldx < xoff + Ci || ldy < yoff + Co || yoff % 2)
        return LB_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    ConvArgs a = {};
    a.x = static_cast<const bf16*>(x); a.ldx = ldx; a.xoff = xoff; a.w = static_cast<const bf16*>(w); a.bias = bias;
    a.y = static_cast<bf16*>(y); a.yf = yf; a.ldy = ldy; a.yoff = yoff;
    a.B = B; a.H = H; a.W = W; a.Ci = Ci; a.Co = Co; a.act = act ? 1 : 0;
    if (g_conv_kernel == 0 || !conv_tc_fits(B, H, W)) return conv_code(conv_mma(a, s));
    if (conv_direct(B, H, W, Ci, Co)) return conv_code(conv_tc(a, s, false));
    void* wp = nullptr;
    cudaError_t e = scratch(&wp, sizeof(bf16) * (size_t)conv_pack_elems(Ci, Co), s);
    if (e != cudaSuccess) return conv_code(e);
    PackArgs p = {};
    p.n = 1;
    p.L[0] = PackLayer{a.w, Ci, Co, static_cast<bf16*>(wp), nullptr, nullptr};
    a.wp = static_cast<bf16*>(wp);
    a.w_late = 1;
    e = conv_pack(p, s);
    if (e == cudaSuccess) e = conv_tc(a, s, true);
    const cudaError_t f = cudaFreeAsync(wp, s);
    return conv_code(e != cudaSuccess ? e : f);
}

int lb_conv3x3_dgrad(const void* gz, const void* w, void* gx, int32_t B, int32_t H, int32_t W, int32_t Ci, int32_t Co,
                     void* stream)
{
    if (!gz || !w || !gx || B < 1 || H < 1 || W < 1 || Ci < 16 || Co < 16 || Ci % 16 || Co % 16) return LB_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const bool tc = g_conv_kernel == 1 && conv_tc_fits(B, H, W);
    void* wt = nullptr;
    cudaError_t e = scratch(&wt, sizeof(bf16) * 9 * (size_t)Ci * Co, s);
    if (e != cudaSuccess) return conv_code(e);
    PackArgs p = {};
    p.n = 1;
    p.L[0] = PackLayer{static_cast<const bf16*>(w), Ci, Co, nullptr, tc ? static_cast<bf16*>(wt) : nullptr,
                       tc ? nullptr : static_cast<bf16*>(wt)};
    ConvArgs a = {};
    a.x = static_cast<const bf16*>(gz); a.ldx = Co;
    (tc ? a.wp : a.w) = static_cast<bf16*>(wt);
    a.w_late = 1;
    a.y = static_cast<bf16*>(gx); a.ldy = Ci;
    a.B = B; a.H = H; a.W = W; a.Ci = Co; a.Co = Ci;
    e = conv_pack(p, s);
    if (e == cudaSuccess) e = tc ? conv_tc(a, s, true) : conv_mma(a, s);
    return conv_code(finish(wt, e, s));
}

int lb_conv3x3_wgrad(const void* x, const void* gz, float* gw, float* gb, int32_t B, int32_t H, int32_t W, int32_t Ci,
                     int32_t Co, void* stream)
{
    if (!x || !gz || !gw || !gb || B < 1 || H < 1 || W < 1 || Ci < 16 || Co < 8 || Ci % 16 || Co % 8) return LB_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    void* part = nullptr;
    const long long room = wgrad_part_elems(B, H, W, Ci, Co);
    cudaError_t e = scratch(&part, sizeof(float) * (size_t)room, s);
    if (e != cudaSuccess) return conv_code(e);
    e = conv_wgrad(s, static_cast<const bf16*>(x), Ci, 0, static_cast<const bf16*>(gz), B, H, W, Ci, Co,
                   static_cast<float*>(part), room, gw, gb, false);
    return conv_code(finish(part, e, s));
}

int lb_conv_release(void)
{
    std::lock_guard<std::mutex> lock(g_pool_mu);
    cudaError_t e = cudaSuccess;
    for (cudaMemPool_t p : g_pools)
        if (p) {
            const cudaError_t f = cudaMemPoolTrimTo(p, 0);
            if (e == cudaSuccess) e = f;
        }
    return conv_code(e);
}

}  // extern "C"
