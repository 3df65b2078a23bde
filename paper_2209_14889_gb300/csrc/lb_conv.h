// lb_conv.h -- the 3x3 convolution kernels of the network (lb_conv.cu): launchers shared with the
// network (lb_unet.cu).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace vlb {
namespace net {

using bf16 = __nv_bfloat16;
constexpr float SLOPE = 0.1f;        // LeakyReLU

// One convolution y[p, o] = b[o] + sum_{t, c} x[p + off_t, c] w[t, o, c], zero padding 1.
struct ConvArgs {
    const bf16* x;          // input, pixel stride ldx, channels at xoff .. xoff + Ci
    long long ldx;
    int xoff;
    const bf16* w;          // [9][Co][Ci] (read by the mma.sync kernel, and by the tcgen05 one without wp)
    const bf16* wp;         // the same weights packed (conv_pack_elems), read by the tcgen05 kernel, or null
    const float* bias;      // [Co] or nullptr
    bf16* y;                // BF16 output (pixel stride ldy, channel offset yoff), or
    float* yf;              // FP32 output
    long long ldy;
    int yoff;
    int B, H, W, Ci, Co;
    int act;                // 1: LeakyReLU
    // optional, with a BF16 output: the LeakyReLU gradient of the layer below, applied to the BF16
    // result by the sign of that layer's stored output ym (pixel stride ldm, channel offset moff)
    const bf16* ym;
    long long ldm;
    int moff;
    // optional, with a BF16 output: a second copy, nearest-upsampled to 2H x 2W (pixel stride ldu,
    // channel offset 0)
    bf16* up;
    long long ldu;
    float* yf2;             // optional, with an FP32 output: a second dense copy (pixel stride ldy)
    int w_late;             // 1: the kernel before this one in the stream writes wp (conv_pack)
};

// BF16 elements of the packed weights of a layer: [Ci / 16][9][2][Co rounded up to 16][8]
inline long long conv_pack_elems(int Ci, int Co) { return (long long)Ci * 9 * ((Co + 15) / 16 * 16); }

// One layer's weights w[9][Co][Ci] in the forms its kernels read; null: not wanted.
struct PackLayer {
    const bf16* w;
    int Ci, Co;
    bf16* fwd;              // packed for the forward pass
    bf16* dgrad;            // w'[8 - t][c][o] = w[t][o][c] packed for the data gradient (Co % 16 == 0)
    bf16* wt;               // w' as [9][Ci][Co]
};
constexpr int PACK_MAX = 16;
struct PackArgs {
    PackLayer L[PACK_MAX];
    int n;
};
cudaError_t conv_pack(const PackArgs& p, cudaStream_t s);

// The tcgen05 kernels index pixels in 32 bits; a larger call takes the mma.sync kernel, which reads the
// weights as they are (a.w) and not packed.
inline bool conv_tc_fits(int B, int H, int W) { return (long long)B * H * W < (1LL << 31); }

// The tcgen05 convolution of a (Ci % 16 == 0, conv_tc_fits).  pdl: the launch may start while the kernel
// before it in the stream finishes (with w_late that kernel may be the one that writes the weights).
// The weights are read packed (a.wp) or, where a.wp is null, as they lie in memory (a.w).
cudaError_t conv_tc(const ConvArgs& a, cudaStream_t s, bool pdl);
// Whether a single call does better with the weights as they lie in memory: packing them costs a launch and
// its scratch (7 us of a call, and 30 at 1024 -> 1024 channels), but bulk copies bring a CTA's packed weights
// in sooner than 16-byte copies of rows that each CTA makes anew.  Few CTAs, or few weights (us, packed and
// not: 8^2, 16 -> 16 channels 34, 26; 16^2, 1024 -> 1024 106, 72; 32^2, 1024 -> 256 78, 51; 75 x 100, 64 -> 96
// 36, 32; 9 x 3000, 32 -> 32 34, 32; beyond, 8 x 128^2, 32 -> 64 42, 44; 256^2, 128 -> 128 51, 57; 2 x 64^2,
// 512 -> 512 81, 123).
bool conv_direct(int B, int H, int W, int Ci, int Co);
// The mma.sync convolution (ym, up and yf2 are not supported).
cudaError_t conv_mma(const ConvArgs& a, cudaStream_t s);

// Weight and bias gradients of one layer from its input x and pre-activation gradient gz (dense
// [P][Co]): gw[9][Co][Ci], gb[Co]; part: scratch of `room` floats (at least 9 Ci Co + Co; with
// wgrad_part_elems floats the reduction is split as far as it pays).  pdl: as for conv_tc.
long long wgrad_part_elems(int B, int H, int W, int Ci, int Co);
cudaError_t conv_wgrad(cudaStream_t s, const bf16* x, long long ldx, int xoff, const bf16* gz, int B, int H, int W,
                       int Ci, int Co, float* part, long long room, float* gw, float* gb, bool pdl);

// the flag that a tcgen05 kernel raises when a bounded wait gave up (nullptr before the first launch)
int* conv_err_flag();

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// launch with or without programmatic stream serialization
template <class K, class... A>
cudaError_t launch_pdl(K kern, dim3 grid, int threads, size_t smem, cudaStream_t s, bool pdl, const A&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace net
}  // namespace vlb
