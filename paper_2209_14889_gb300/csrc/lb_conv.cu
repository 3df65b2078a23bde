// lb_conv.cu -- 3x3 convolutions on NHWC BF16 activations with FP32 accumulation (the network of
// the learned stepper) as implicit GEMMs: forward passes and data gradients with the pixels as M, the
// output channels as N and K = 9 Ci, weight gradients with the input channels as M, the output channels
// as N and the pixels as K.
#include <algorithm>
#include <atomic>
#include <cstdint>

#include "lb_conv.h"
#include "lb_internal.h"

namespace vlb {
namespace net {

namespace {

// ------------------------------------------------------------------ tensor-core primitives

__device__ __forceinline__ unsigned smem_u32(const void* p)
{
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void ldsm_x4(unsigned (&r)[4], const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p)));
}
// D += A (16x16, row) * B (16x8, col); BF16 inputs, FP32 accumulators
__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ------------------------------------------------------------------ mma.sync convolution

constexpr int CT_H = 8, CT_W = 16;              // output tile: 8 rows x 16 pixels (4 warps x 2 rows)
constexpr int CT_IH = CT_H + 2, CT_IW = CT_W + 2;
constexpr int CT_CO = 64;                       // output channels per CTA
constexpr int PS = 24;                          // shared row of 16 channels + 8 pad (48 bytes)

// MINB CTAs per SM: 4 leave a thread 120 registers, 5 (what the compiler chooses by itself) 96.  conv_mma takes
// the larger number where it saves a wave of CTAs, and the registers where it does not.
// ODD: a BF16 output at an odd pixel stride or address, stored value by value.
template <int MINB, bool ODD>
__global__ void __launch_bounds__(128, MINB) k_conv3x3(const ConvArgs a)
{
    __shared__ __align__(16) bf16 sx[CT_IH * CT_IW * PS];
    __shared__ __align__(16) bf16 sw[9 * CT_CO * PS];
    const int n_cot = (a.Co + CT_CO - 1) / CT_CO;
    const int b = blockIdx.z / n_cot, co0 = (blockIdx.z % n_cot) * CT_CO;
    const int tx0 = blockIdx.x * CT_W, ty0 = blockIdx.y * CT_H;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float acc[2][8][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[i][j][k] = 0.f;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);

    for (int c0 = 0; c0 < a.Ci; c0 += 16) {
        for (int q = tid; q < CT_IH * CT_IW * 2; q += 128) {
            const int p = q >> 1, h = q & 1;
            const int py = p / CT_IW, px = p - py * CT_IW;
            const int gy = ty0 - 1 + py, gx = tx0 - 1 + px;
            uint4 v = zero;
            if (gy >= 0 && gy < a.H && gx >= 0 && gx < a.W)
                v = *reinterpret_cast<const uint4*>(a.x + ((long long)(b * a.H + gy) * a.W + gx) * a.ldx + a.xoff + c0 +
                                                    h * 8);
            *reinterpret_cast<uint4*>(sx + p * PS + h * 8) = v;
        }
        for (int q = tid; q < 9 * CT_CO * 2; q += 128) {
            const int t = q / (CT_CO * 2), r = q - t * (CT_CO * 2);
            const int co = r >> 1, h = r & 1;
            uint4 v = zero;
            if (co0 + co < a.Co)
                v = *reinterpret_cast<const uint4*>(a.w + ((long long)t * a.Co + co0 + co) * a.Ci + c0 + h * 8);
            *reinterpret_cast<uint4*>(sw + (t * CT_CO + co) * PS + h * 8) = v;
        }
        __syncthreads();
#pragma unroll 1
        for (int t = 0; t < 9; ++t) {
            const int dy = t / 3 - 1, dx = t % 3 - 1;
            unsigned A[2][4];
#pragma unroll
            for (int mi = 0; mi < 2; ++mi) {
                const int orow = warp * 2 + mi;
                const int pix = (lane & 7) + ((lane >> 3) & 1) * 8;
                const int sp = (orow + 1 + dy) * CT_IW + (pix + 1 + dx);
                ldsm_x4(A[mi], sx + sp * PS + (lane >> 4) * 8);
            }
#pragma unroll
            for (int nj = 0; nj < 8; nj += 2) {
                unsigned Bf[4];
                const int n = nj * 8 + (lane & 7) + (lane >> 4) * 8;
                ldsm_x4(Bf, sw + (t * CT_CO + n) * PS + ((lane >> 3) & 1) * 8);
#pragma unroll
                for (int mi = 0; mi < 2; ++mi) {
                    mma_bf16(acc[mi][nj], A[mi], Bf[0], Bf[1]);
                    mma_bf16(acc[mi][nj + 1], A[mi], Bf[2], Bf[3]);
                }
            }
        }
        __syncthreads();
    }

    // epilogue: bias, activation, store (thread holds rows g, g+8 and channel pairs 2t, 2t+1)
    const int g = lane >> 2, tq = lane & 3;
#pragma unroll
    for (int mi = 0; mi < 2; ++mi) {
        const int gy = ty0 + warp * 2 + mi;
        if (gy >= a.H) continue;
#pragma unroll
        for (int nj = 0; nj < 8; ++nj) {
            const int co = co0 + nj * 8 + 2 * tq;
            if (co >= a.Co) continue;
            const float b0 = a.bias ? a.bias[co] : 0.f, b1 = a.bias ? a.bias[co + 1] : 0.f;
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const int gx = tx0 + g + 8 * hh;
                if (gx >= a.W) continue;
                float v0 = acc[mi][nj][2 * hh] + b0, v1 = acc[mi][nj][2 * hh + 1] + b1;
                if (a.act) {
                    v0 = v0 > 0.f ? v0 : SLOPE * v0;
                    v1 = v1 > 0.f ? v1 : SLOPE * v1;
                }
                const long long o = ((long long)(b * a.H + gy) * a.W + gx) * a.ldy + a.yoff + co;
                if (a.yf) {
                    a.yf[o] = v0;
                    a.yf[o + 1] = v1;
                } else {
                    const __nv_bfloat162 r = __floats2bfloat162_rn(v0, v1);
                    if (!ODD) {
                        *reinterpret_cast<__nv_bfloat162*>(a.y + o) = r;
                    } else {
                        a.y[o] = r.x;
                        a.y[o + 1] = r.y;
                    }
                }
            }
        }
    }
}

// ------------------------------------------------------------------ tcgen05 convolution
//
// A CTA computes 128 MT consecutive positions (MT MMA tiles of M = 128) of a position space in which
// the taps are constant offsets, for `cop` output channels (N).  The positions come in two forms:
//   flat   (W <= 128): Q = (b (H + 1) + y) (W + 1) + x; the column x = W and the row y = H are zeros
//          that serve as the padding of their neighbours on both sides, so only 1 / (W + 1) of the
//          positions are padding, whatever the image's size; the taps reach W + 2 positions around;
//   tiles  (W > 128): 4 MT rows of 32 positions, 30 of them output columns (columns 30, 31 of a row
//          run into the next one and are not stored), where the flat form's halo of 2 (W + 2)
//          positions would outweigh the tile.
// Either way a tap reads the 128 consecutive staged positions that start at (1 + dy) pitch + 1 + dx.
// One chunk of 16 input channels is 9 MT MMAs of K = 16, in the same order for every geometry (chunk,
// then tap), so results do not depend on it.  Operands in the canonical K-major layout without
// swizzle: input [k-halves][positions][8], weights [chunks][9 taps][2 k-halves][cop][8]; 8-row groups
// 128 bytes apart.
//
// Eight warps copy the input (cp.async; the pixels of the positions in a table formed once), one warp
// the weights (bulk copies of the packed layout, conv_pack), one warp issues the MMAs.  A stage holds
// cw = 1, 2 or 4 chunks, so that a copy instruction covers 32 to 128 contiguous bytes of a pixel;
// each of up to 16 stages has a barrier for its input, its weights and its release by the MMAs that
// read it (tcgen05.commit).  The eight copying warps then store the result, two per quarter of the
// tensor memory's lanes.
//
// What bounds it: the 128 x 16 input operand of every MMA is read from shared memory (4 KB, 32 cycles
// against 16 of tensor work at 32 channels); the copies of the input; at few CTAs (the 1/4 and 1/8
// resolution layers) the latency of one CTA's chain, which is why all copies are issued ahead and the
// channels are split until most SMs have a CTA.

// shared-memory matrix descriptor: start address, leading (K-direction core-matrix) and stride
// (8-row group) byte offsets, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t tc_desc(unsigned saddr, unsigned lbo, unsigned sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);   // version 1, no swizzle
}

__device__ __forceinline__ void cp_async16(unsigned sdst, const void* gsrc, int src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sdst), "l"(gsrc), "r"(src_bytes) : "memory");
}
// the barrier's count drops by one when all copies issued so far by this thread have landed
__device__ __forceinline__ void cp_async_arrive(uint64_t* mb)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(mb)) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void bulk_copy(unsigned sdst, const void* gsrc, unsigned bytes, uint64_t* mb)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(sdst),
                 "l"(gsrc), "r"(bytes), "r"(smem_u32(mb))
                 : "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t* mb, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mb)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* mb, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mb)), "r"(bytes) : "memory");
}
// bounded wait for the phase of parity `parity` of an mbarrier; false if it gave up
__device__ __forceinline__ bool mbar_wait(uint64_t* mb, unsigned parity)
{
    unsigned done = 0;
    for (long it = 0; it < (1L << 20) && !done; ++it) {
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(smem_u32(mb)), "r"(parity)
            : "memory");
    }
    return done != 0;
}
__device__ __forceinline__ void tc_commit(uint64_t* mb)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mb)) : "memory");
}
// One lane issues the MMAs, but the whole warp runs the loop around them with warp-uniform operands: in
// a branch of one thread the descriptors go through that thread's registers and each MMA took 130 to 160
// cycles to issue, against 32 + N / 4 this way (measured, N = 16 .. 128: the operands' shared memory).
__device__ __forceinline__ unsigned elect_one()
{
    unsigned l;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(l));
    return l;
}
__device__ __forceinline__ void tc_mma(unsigned d, uint64_t ad, uint64_t bd, uint32_t idesc, int acc, unsigned lead)
{
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc), "r"(lead));
}
__device__ __forceinline__ void tc_ld16(unsigned (&v)[16], unsigned taddr)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
        "%13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tc_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 32 bytes to global memory (32-byte aligned): a whole sector per lane
__device__ __forceinline__ void st32(void* p, const unsigned (&v)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
                 "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

constexpr int TC_COPY = 256;                     // threads of the 8 copying and storing warps
constexpr int TC_THREADS = TC_COPY + 64;         // and the MMA warp and the weights (bias) warp
constexpr int TC_SLOTS = 16;                     // most stages
constexpr int TC_HEAD = 1024;                    // shared bytes of the barriers and the bias

// division of 0 <= n < 2^31 by a constant d >= 1 by a multiplication and a shift (Granlund and Montgomery,
// Division by invariant integers using multiplication, 1994): n / d = ((n m >> 32) + n) >> s with 2^s >= d
struct FastDiv {
    unsigned m, s, d;
    FastDiv() = default;
    explicit FastDiv(unsigned d_) : d(d_)
    {
        for (s = 0; (1u << s) < d && s < 31; ++s) {
        }
        m = (unsigned)((((1ull << s) - d) << 32) / d + 1);       // 2^32 (2^s - d) / d, rounded up
    }
    __device__ __forceinline__ unsigned div(unsigned n) const { return (unsigned)(((unsigned long long)__umulhi(n, m) + n) >> s); }
};

struct ConvGeo {
    int flat, pitch, npix;                       // npix: staged positions
    int cop, slots, tx, ty;                      // channels per CTA, stages, tile grid (tiles form)
    int cw, lgh;                                 // chunks per stage, log2 of its k-halves
    int cpk;                                     // channels of the packed weights
    unsigned ncol;                               // tensor-memory columns (a power of two >= 32)
    FastDiv d0, d1;                              // flat: by pitch, by H + 1; tiles: by tx, by tx ty
};

// shared state of a tcgen05 kernel ahead of its stages
struct TcShared {
    uint64_t xfull[TC_SLOTS], wfull[TC_SLOTS], empty[TC_SLOTS], done;
    unsigned tmem;
    int fail;
    float4 bias[32];
};
static_assert(sizeof(TcShared) <= TC_HEAD, "barriers fit ahead of the stages");

// output position -> pixel (b, y, x); false where there is none
template <int MT>
__device__ __forceinline__ bool out_pixel(const ConvArgs& a, const ConvGeo& g, int mt, int m, int& b, int& y, int& x)
{
    if (g.flat) {
        const int Q = (int)blockIdx.x * (128 * MT) + 128 * mt + m;
        const int row = (int)g.d0.div((unsigned)Q);
        x = Q - row * g.pitch;
        b = (int)g.d1.div((unsigned)row);
        y = row - b * (a.H + 1);
        return x < a.W && y < a.H && b < a.B;
    }
    b = (int)g.d1.div(blockIdx.x);
    const int r = (int)blockIdx.x - b * g.tx * g.ty;
    const int ty = (int)g.d0.div((unsigned)r);
    const int c = m & 31;
    y = ty * (4 * MT) + 4 * mt + (m >> 5);
    x = (r - ty * g.tx) * 30 + c;
    return c < 30 && x < a.W && y < a.H;
}

// pixel at staged position p, or -1 where it is padding (there are fewer than 2^31 pixels)
template <int MT>
__device__ __forceinline__ int in_pixel(const ConvArgs& a, const ConvGeo& g, int p)
{
    int b, y, x;
    if (g.flat) {
        const int Q = (int)blockIdx.x * (128 * MT) - g.pitch - 1 + p;
        if (Q < 0 || p >= 128 * MT + 2 * g.pitch + 2) return -1;
        const int row = (int)g.d0.div((unsigned)Q);
        x = Q - row * g.pitch;
        b = (int)g.d1.div((unsigned)row);
        y = row - b * (a.H + 1);
        if (b >= a.B) return -1;
    } else {
        b = (int)g.d1.div(blockIdx.x);
        const int r = (int)blockIdx.x - b * g.tx * g.ty;
        const int ty = (int)g.d0.div((unsigned)r);
        y = ty * (4 * MT) - 1 + (p >> 5);
        x = (r - ty * g.tx) * 30 - 1 + (p & 31);
        if (p >= (4 * MT + 2) * 32 || y < 0 || x < 0) return -1;
    }
    if (x >= a.W || y >= a.H) return -1;
    return (b * a.H + y) * a.W + x;
}

// DIRECT: the weights come as they lie in memory (a.w), by the copying warps
template <int MT, bool DIRECT>
__global__ void __launch_bounds__(TC_THREADS) k_conv_tc(const __grid_constant__ ConvArgs a, const __grid_constant__ ConvGeo g,
                                                        int* err)
{
    extern __shared__ __align__(128) unsigned char smem[];
    TcShared& S = *reinterpret_cast<TcShared*>(smem);
    int* const spix = reinterpret_cast<int*>(smem + TC_HEAD);        // pixels of the staged positions
    const int xbytes = g.npix * 32 * g.cw, sbytes = xbytes + 288 * g.cop * g.cw;
    const unsigned stage0 = smem_u32(smem) + TC_HEAD + (unsigned)(g.npix * 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int co0 = blockIdx.y * g.cop;
    const int nstage = a.Ci / (16 * g.cw), slots = g.slots;

    if (tid == 0) {
        for (int s = 0; s < slots; ++s) {
            mbar_init(&S.xfull[s], TC_COPY);
            mbar_init(&S.wfull[s], 1);
            mbar_init(&S.empty[s], 1);
        }
        mbar_init(&S.done, 1);
        S.fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == TC_COPY / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem)),
                     "r"(g.ncol));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    for (int p = tid; p < g.npix; p += TC_THREADS) spix[p] = in_pixel<MT>(a, g, p);
    if (tid < 128) reinterpret_cast<float*>(S.bias)[tid] = a.bias && tid < g.cop && co0 + tid < a.Co ? a.bias[co0 + tid] : 0.f;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = S.tmem;

    bool ok = true;
    if (warp < TC_COPY / 32) {
        // ---- input: 16-byte units (position, k-half), the k-halves of a position side by side
        const int h = tid & ((1 << g.lgh) - 1), p0 = tid >> g.lgh, step = TC_COPY >> g.lgh;
        pdl_wait();                       // the input is the result of the kernel before this one
        for (int k = 0; k < nstage && ok; ++k) {
            const int s = k % slots;
            if (k >= slots) ok = mbar_wait(&S.empty[s], (unsigned)((k / slots - 1) & 1));
            if (!ok) break;
            if (DIRECT) {
                // the weights as they lie in memory: a row (tap, output channel) of the stage's channels is
                // one run of 16-byte units
                const int units = min(g.cop, a.Co - co0) << g.lgh;
                for (int v = tid; v < units; v += TC_COPY) {
                    const int hw = v & ((1 << g.lgh) - 1), co = v >> g.lgh;
                    const bf16* src = a.w + (long long)(co0 + co) * a.Ci + 16 * g.cw * k + 8 * hw;
                    const unsigned d = stage0 + (unsigned)(s * sbytes + xbytes + (((hw >> 1) * 18 + (hw & 1)) * g.cop + co) * 16);
#pragma unroll
                    for (int t = 0; t < 9; ++t)
                        cp_async16(d + (unsigned)(t * 2 * g.cop * 16), src + (long long)t * a.Co * a.Ci, 16);
                }
            }
            const unsigned dst = stage0 + (unsigned)(s * sbytes + h * g.npix * 16);
            const bf16* base = a.x + a.xoff + 16 * g.cw * k + 8 * h;
#pragma unroll 4
            for (int p = p0; p < g.npix; p += step) {
                const int pix = spix[p];
                cp_async16(dst + (unsigned)(p * 16), pix >= 0 ? base + (long long)pix * a.ldx : a.x, pix >= 0 ? 16 : 0);
            }
            cp_async_arrive(&S.xfull[s]);
        }
        pdl_trigger();
    } else if (warp == TC_COPY / 32 + 1) {
        // ---- weights: 18 bulk copies (tap, k-half) of the CTA's channels per chunk
        const unsigned nb = (unsigned)min(g.cop, g.cpk - co0) * 16u;
        int issued = 0;
        if (!DIRECT && a.w_late) pdl_wait();
        for (int k = 0; !DIRECT && k < nstage && ok; ++k) {
            const int s = k % slots;
            if (k >= slots) ok = __all_sync(0xffffffffu, mbar_wait(&S.empty[s], (unsigned)((k / slots - 1) & 1)));
            if (!ok) break;
            if (lane == 0) mbar_expect_tx(&S.wfull[s], 18u * (unsigned)g.cw * nb);
            __syncwarp();
            for (int q = lane; q < 18 * g.cw; q += 32)
                bulk_copy(stage0 + (unsigned)(s * sbytes + xbytes + q * g.cop * 16),
                          a.wp + (((long long)k * g.cw * 18 + q) * g.cpk + co0) * 8, nb, &S.wfull[s]);
            issued = k + 1;
        }
        // the CTA does not end with a weights copy in flight, whatever happened above
        for (int k = max(0, issued - slots); k < issued; ++k)
            mbar_wait(&S.wfull[k % slots], (unsigned)((k / slots) & 1));
    } else {
        // ---- MMAs
        const unsigned lead = elect_one();
        const uint32_t idesc =
            (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(g.cop >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        for (int k = 0; k < nstage && ok; ++k) {
            const int s = k % slots;
            const unsigned par = (unsigned)((k / slots) & 1);
            ok = __all_sync(0xffffffffu, mbar_wait(&S.xfull[s], par) && (DIRECT || mbar_wait(&S.wfull[s], par)));
            if (!ok) break;
            // the input was written through the generic proxy, the tensor core reads through the
            // asynchronous one
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // descriptors of the tap (-1, -1); their addresses count 16 bytes: positions and weights
            const unsigned sx = stage0 + (unsigned)(s * sbytes);
            uint64_t ad = tc_desc(sx, (unsigned)(g.npix * 16), 128);
            uint64_t bd = tc_desc(sx + (unsigned)xbytes, (unsigned)(g.cop * 16), 128);
            for (int kk = 0; kk < g.cw; ++kk) {
#pragma unroll
                for (int t = 0; t < 9; ++t) {
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
                        tc_mma(tmem + (unsigned)(mt * g.cop), ad + (unsigned)((t / 3) * g.pitch + t % 3 + 128 * mt),
                               bd + (unsigned)(t * 2 * g.cop), idesc, (k > 0 || kk > 0 || t > 0) ? 1 : 0, lead);
                }
                ad += (unsigned)(2 * g.npix);
                bd += (unsigned)(18 * g.cop);
            }
            if (lead) tc_commit(&S.empty[s]);
        }
        if (ok && lead) tc_commit(&S.done);
    }
    if (!ok) S.fail = 1;

    if (warp < TC_COPY / 32) {
        if (ok) ok = mbar_wait(&S.done, 0);
        if (!ok) S.fail = 1;
        cp_async_wait_all();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok) {
            // warp w holds the positions 32 (w % 4) .. of each tile, the columns are the channels co0 ..;
            // blocks of 16 channels of a tile, every second one, two at a time
            const int m = tid & 127, nj = g.cop / 16, nblk = MT * nj;
            const unsigned lane0 = tmem + ((unsigned)(warp & 3) << 21);
            for (int q0 = warp >> 2; q0 < nblk; q0 += 4) {
                __syncwarp();               // the lanes that stored nothing and the others
                unsigned v[2][16];
                const int q1 = q0 + 2;
                tc_ld16(v[0], lane0 + (unsigned)((q0 / nj) * g.cop + (q0 % nj) * 16));
                if (q1 < nblk) tc_ld16(v[1], lane0 + (unsigned)((q1 / nj) * g.cop + (q1 % nj) * 16));
                tc_ld_wait();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int q = h ? q1 : q0;
                    if (q >= nblk) break;
                    const int mt = q / nj, j = (q - mt * nj) * 16;
                    int b, y, x;
                    if (!out_pixel<MT>(a, g, mt, m, b, y, x)) continue;
                    const long long pix = ((long long)b * a.H + y) * a.W + x;
                    const long long o = pix * a.ldy + a.yoff + co0 + j;
                    float f[16];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float4 bi = S.bias[j / 4 + e];
                        f[4 * e] = __uint_as_float(v[h][4 * e]) + bi.x;
                        f[4 * e + 1] = __uint_as_float(v[h][4 * e + 1]) + bi.y;
                        f[4 * e + 2] = __uint_as_float(v[h][4 * e + 2]) + bi.z;
                        f[4 * e + 3] = __uint_as_float(v[h][4 * e + 3]) + bi.w;
                    }
                    if (a.act) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) f[e] = fmaxf(f[e], SLOPE * f[e]);      // LeakyReLU, 0 < SLOPE < 1
                    }
                    // stores of a whole sector where the address allows, in eights (the last block of a
                    // channel count that is no multiple of 16 has one, and every second pixel starts
                    // between sectors), else value by value: 3 x 441 x 395, 32 -> 88 channels 268 us value
                    // by value, 99 in eights
                    const int n8 = min(2, (a.Co - co0 - j) / 8);
                    if (a.yf) {
                        const unsigned(*w)[8] = reinterpret_cast<const unsigned(*)[8]>(f);
                        const bool sect = (((uintptr_t)(a.yf + o) | (a.yf2 ? (uintptr_t)(a.yf2 + o) : 0)) & 31) == 0;
#pragma unroll
                        for (int q8 = 0; q8 < 2; ++q8) {
                            if (q8 >= n8) break;
                            if (sect) {
                                st32(a.yf + o + 8 * q8, w[q8]);
                                if (a.yf2) st32(a.yf2 + o + 8 * q8, w[q8]);
                            } else {
#pragma unroll
                                for (int e = 8 * q8; e < 8 * q8 + 8; ++e) {
                                    a.yf[o + e] = f[e];
                                    if (a.yf2) a.yf2[o + e] = f[e];
                                }
                            }
                        }
                        continue;
                    }
                    __nv_bfloat162 r[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) r[e] = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
                    if (a.ym) {                     // the gradient through the layer below's LeakyReLU
                        const uint4* mp = reinterpret_cast<const uint4*>(a.ym + pix * a.ldm + a.moff + co0 + j);
                        const uint4 m4[2] = {mp[0], mp[1]};     // not __ldg: a launch before wrote them
                        const __nv_bfloat162* mv = reinterpret_cast<const __nv_bfloat162*>(m4);
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const float2 gg = __bfloat1622float2(r[e]), mm = __bfloat1622float2(mv[e]);
                            r[e] = __floats2bfloat162_rn(mm.x > 0.f ? gg.x : SLOPE * gg.x, mm.y > 0.f ? gg.y : SLOPE * gg.y);
                        }
                    }
                    const unsigned(&w)[8] = *reinterpret_cast<const unsigned(*)[8]>(r);
                    if (n8 == 2 && ((uintptr_t)(a.y + o) & 31) == 0) {
                        st32(a.y + o, w);
                    } else if (((uintptr_t)(a.y + o) & 15) == 0) {
                        const uint4* v8 = reinterpret_cast<const uint4*>(r);
                        if (n8 > 0) reinterpret_cast<uint4*>(a.y + o)[0] = v8[0];
                        if (n8 > 1) reinterpret_cast<uint4*>(a.y + o)[1] = v8[1];
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            if (e < 8 * n8) a.y[o + e] = e & 1 ? r[e >> 1].y : r[e >> 1].x;
                    }
                    if (a.up) {                     // the network's own buffers: whole blocks, aligned
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            st32(a.up + (((long long)b * 2 * a.H + 2 * y + (u >> 1)) * 2 * a.W + 2 * x + (u & 1)) * a.ldu + co0 + j,
                                 w);
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (S.fail && tid == 0) atomicExch(err, 1);
    if (warp == TC_COPY / 32) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(g.ncol));
    }
}

// ------------------------------------------------------------------ weight gradient
//
// gw[t][co][ci] = sum over pixels of gz[p][co] x[p + off_t][ci] on the tensor cores: M = input channels
// (up to 128 per CTA), N = (dx, output channel), up to 3 x 48, K = pixels q = p + dx of an input row; one
// accumulator of N columns per dy (3 N <= 432 of the 512 tensor-memory columns), so one pass over the
// pixels serves all nine taps.  The channels are the contiguous index of both operands, so they are read
// MN-major: [channel group of 8][position][8].  The gradient row is staged three times, shifted by dx,
// as three runs of channel groups.
// A CTA takes units of up to RB rows of a 32-column strip, every S-th unit: stage j of a unit brings
// gradient row y0 - 1 + j and, from j = 2, input row r = y0 + j - 2, whose 6 MMAs (2 x 16 positions,
// 3 dy) then read the gradient rows r - dy of the stages j - 2 .. j.  Up to 16 stages are in flight; a
// stage is released by the MMAs that read it last and by the warp that adds the gradient rows for the
// bias.  Each CTA writes one partial sum, k_sum_parts adds the S partials in a fixed order.
// What bounds it: the M = 128 operand of an MMA takes 32 cycles to read from shared memory, whatever its
// N (at few input channels most of its rows are not used, which costs nothing more), so the taps of a
// row share it: N = 96 takes 56 cycles where three of N = 32 take 3 x 40.

struct WgradArgs {
    const bf16* x;          // layer input (pixel stride ldx, offset xoff)
    long long ldx;
    int xoff;
    const bf16* gz;         // gradient at the layer's pre-activation output, dense [P][Co]
    float* part;            // [S][n] partial sums: [9][Ci][Co], then the bias [Co] (32-byte aligned)
    int B, H, W, Ci, Co;
};

struct WgradGeo {
    int cib, cob;           // channels per CTA
    int RB, strips, rbs;    // rows per unit, strips per row, units per strip
    int units, slots;
    unsigned ncol;
    long long n;            // values of a partial sum
};

constexpr int WG_P = 32;                         // positions of a staged row
constexpr int WG_NMAX = 48;

__global__ void __launch_bounds__(TC_THREADS) k_wgrad_tc(const __grid_constant__ WgradArgs a,
                                                         const __grid_constant__ WgradGeo g, int* err)
{
    extern __shared__ __align__(128) unsigned char smem[];
    TcShared& S = *reinterpret_cast<TcShared*>(smem);
    const int zg = g.cob / 8;
    const int xbytes = g.cib / 8 * WG_P * 16, sbytes = xbytes + 3 * zg * WG_P * 16;
    const unsigned stage0 = smem_u32(smem) + TC_HEAD;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ci0 = blockIdx.y * g.cib, co0 = blockIdx.z * g.cob;
    const int xg = min(g.cib, a.Ci - ci0) / 8;   // input channel groups of this CTA
    const int slots = g.slots;

    if (tid == 0) {
        for (int s = 0; s < slots; ++s) {
            mbar_init(&S.xfull[s], TC_COPY);
            mbar_init(&S.empty[s], 2);
        }
        mbar_init(&S.done, 1);
        S.fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == TC_COPY / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem)),
                     "r"(g.ncol));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = S.tmem;
    const int per = g.strips * g.rbs;

    bool ok = true;
    if (warp < TC_COPY / 32) {
        // ---- rows: 16-byte units (position, channel group), the channels of a position side by side
        constexpr int NX = 2, NZ = 3;       // units per thread: 16 x 32 / 256, 18 x 32 / 256
        int xp[NX], xd[NX], zp[NZ], zd[NZ];
        long long xs[NX], zs[NZ];
#pragma unroll
        for (int i = 0; i < NX; ++i) {
            const int u = tid + TC_COPY * i, p = u / xg, q = u - p * xg;
            xp[i] = p < WG_P ? p : -1;
            xd[i] = (q * WG_P + p) * 16;
            xs[i] = (long long)p * a.ldx + a.xoff + ci0 + 8 * q;
        }
#pragma unroll
        for (int i = 0; i < NZ; ++i) {
            // (dx, position, group): position q of copy dx holds the gradient at column q - dx
            const int u = tid + TC_COPY * i, r = u / zg, q = u - r * zg, dx = r / WG_P - 1, p = r % WG_P;
            const bool in = dx <= 1 && co0 + 8 * q < a.Co;
            zp[i] = dx <= 1 ? (in ? p - dx : -2) : -3;
            zd[i] = xbytes + (((dx + 1) * zg + q) * WG_P + p) * 16;
            zs[i] = (long long)(p - dx) * a.Co + co0 + 8 * q;
        }
        pdl_wait();
        int s = 0;
        unsigned par = 1;                   // the first round finds the stages free
        const long long zrow = (long long)a.W * a.Co, xrow = (long long)a.W * a.ldx;
        for (int u = blockIdx.x; u < g.units && ok; u += gridDim.x) {
            const int b = u / per, r = u - b * per;
            const int x0 = (r / g.rbs) * WG_P, y0 = (r % g.rbs) * g.RB;
            const int rows = min(g.RB, a.H - y0);
            // this thread's columns of the strip: inside the image or not
            bool xin[NX], zin[NZ];
#pragma unroll
            for (int i = 0; i < NX; ++i) xin[i] = x0 + xp[i] < a.W;
#pragma unroll
            for (int i = 0; i < NZ; ++i) zin[i] = zp[i] > -2 && x0 + zp[i] >= 0 && x0 + zp[i] < a.W;
            const bf16* bz = a.gz + (((long long)b * a.H + y0 - 1) * a.W + x0) * a.Co;
            const bf16* bx = a.x + (((long long)b * a.H + y0 - 2) * a.W + x0) * a.ldx;
            for (int j = 0; j < rows + 2; ++j, bz += zrow, bx += xrow) {
                ok = mbar_wait(&S.empty[s], par);
                if (!ok) break;
                const unsigned dst = stage0 + (unsigned)(s * sbytes);
                const bool rowz = y0 - 1 + j >= 0 && y0 - 1 + j < a.H;
#pragma unroll
                for (int i = 0; i < NZ; ++i) {
                    if (zp[i] == -3) continue;
                    const bool in = rowz && zin[i];
                    cp_async16(dst + (unsigned)zd[i], in ? bz + zs[i] : a.gz, in ? 16 : 0);
                }
                if (j >= 2) {
#pragma unroll
                    for (int i = 0; i < NX; ++i) {
                        if (xp[i] < 0) continue;
                        cp_async16(dst + (unsigned)xd[i], xin[i] ? bx + xs[i] : a.x, xin[i] ? 16 : 0);
                    }
                }
                cp_async_arrive(&S.xfull[s]);
                if (++s == slots) {
                    s = 0;
                    par ^= 1u;
                }
            }
        }
        pdl_trigger();
    } else if (warp == TC_COPY / 32 + 1) {
        // ---- bias: the gradient rows added up, one position per lane
        float acc[WG_NMAX];
#pragma unroll
        for (int e = 0; e < WG_NMAX; ++e) acc[e] = 0.f;
        int s = 0;
        unsigned par = 0;
        for (int u = blockIdx.x; u < g.units && ok; u += gridDim.x) {
            const int r = u % per;
            const int rows = min(g.RB, a.H - (r % g.rbs) * g.RB);
            for (int j = 0; j < rows + 2; ++j) {
                // every stage is waited for, so that this warp's arrival belongs to the stage's own phase
                ok = __all_sync(0xffffffffu, mbar_wait(&S.xfull[s], par));
                if (!ok) break;
                if (j >= 1 && j <= rows && blockIdx.y == 0) {       // the unit's own rows, unshifted
                    const unsigned char* z = smem + TC_HEAD + s * sbytes + xbytes + (zg * WG_P + lane) * 16;
#pragma unroll
                    for (int q = 0; q < WG_NMAX / 8; ++q) {
                        if (q >= zg) break;
                        const uint4 v = *reinterpret_cast<const uint4*>(z + q * WG_P * 16);
                        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 f = __bfloat1622float2(h[e]);
                            acc[8 * q + 2 * e] += f.x;
                            acc[8 * q + 2 * e + 1] += f.y;
                        }
                    }
                }
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&S.empty[s])) : "memory");
                if (++s == slots) {
                    s = 0;
                    par ^= 1u;
                }
            }
        }
        if (ok && blockIdx.y == 0) {
            pdl_wait();             // the partial sums' buffer is the former reduction's
#pragma unroll
            for (int e = 0; e < WG_NMAX; ++e) {
                float v = acc[e];
                for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                if (lane == 0 && e < g.cob && co0 + e < a.Co)
                    a.part[blockIdx.x * g.n + 9LL * a.Co * a.Ci + co0 + e] = v;
            }
        }
    } else {
        // ---- MMAs, both operands MN-major
        const unsigned lead = elect_one();
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                               ((uint32_t)(3 * g.cob >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        int s = 0, s1 = 0, s2 = 0, acc = 0;         // this stage and the two before it
        unsigned par = 0;
        for (int u = blockIdx.x; u < g.units && ok; u += gridDim.x) {
            const int r = u % per;
            const int rows = min(g.RB, a.H - (r % g.rbs) * g.RB);
            for (int j = 0; j < rows + 2; ++j) {
                ok = __all_sync(0xffffffffu, mbar_wait(&S.xfull[s], par));
                if (!ok) break;
                const int sn = s + 1 == slots ? 0 : s + 1;
                if (j < 2) {
                    s2 = s1;
                    s1 = s;
                    if (sn == 0) par ^= 1u;
                    s = sn;
                    continue;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t ad = tc_desc(stage0 + (unsigned)(s * sbytes), 128, WG_P * 16);
#pragma unroll
                for (int dy = -1; dy <= 1; ++dy) {          // gradient row r - dy: 1 + dy stages back
                    const int sz = dy < 0 ? s : (dy == 0 ? s1 : s2);
                    const uint64_t bd = tc_desc(stage0 + (unsigned)(sz * sbytes + xbytes), 128, WG_P * 16);
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks)
                        tc_mma(tmem + (unsigned)((dy + 1) * 3 * g.cob), ad + (unsigned)(16 * ks), bd + (unsigned)(16 * ks), idesc,
                               ks > 0 ? 1 : acc, lead);
                }
                acc = 1;
                if (lead) {
                    tc_commit(&S.empty[s2]);
                    if (j == rows + 1) {
                        tc_commit(&S.empty[s1]);
                        tc_commit(&S.empty[s]);
                    }
                }
                s2 = s1;
                s1 = s;
                if (sn == 0) par ^= 1u;
                s = sn;
            }
        }
        if (ok && lead) tc_commit(&S.done);
    }
    if (!ok) S.fail = 1;

    if (warp < TC_COPY / 32) {
        if (ok) ok = mbar_wait(&S.done, 0);
        if (!ok) S.fail = 1;
        cp_async_wait_all();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok) {
            // warp w holds the input channels 32 (w % 4) .., the columns are the output channels co0 .. of
            // each tap; blocks of 16 of them, every second one, two at a time
            const int m = tid & 127, nj = g.cob / 16, nblk = 9 * nj;
            const bool valid = m < 8 * xg;
            const unsigned lane0 = tmem + ((unsigned)(warp & 3) << 21);
            // a lane holds 16 output channels of its input channel: two whole sectors of [9][Ci][Co] (one
            // store per value, along the input channels, took 6 to 10 us of 18 to 38)
            float* out = a.part + blockIdx.x * g.n + (long long)(ci0 + m) * a.Co;
            for (int q0 = warp >> 2; q0 < nblk; q0 += 4) {
                __syncwarp();               // the lanes that stored nothing and the others
                unsigned v[2][16];
                tc_ld16(v[0], lane0 + (unsigned)(q0 * 16));
                if (q0 + 2 < nblk) tc_ld16(v[1], lane0 + (unsigned)((q0 + 2) * 16));
                tc_ld_wait();
                if (!valid) continue;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int q = q0 + 2 * h;
                    if (q >= nblk) break;
                    const int t = q / nj, co = co0 + (q - t * nj) * 16;
                    float* o = out + (long long)t * a.Ci * a.Co + co;
                    const unsigned(&w)[2][8] = *reinterpret_cast<const unsigned(*)[2][8]>(v[h]);
                    if (co < a.Co) st32(o, w[0]);
                    if (co + 8 < a.Co) st32(o + 8, w[1]);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (S.fail && tid == 0) atomicExch(err, 1);
    if (warp == TC_COPY / 32) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(g.ncol));
    }
}

// Sum of S partial arrays of n floats (n a multiple of 4): eight threads per float4, each every eighth
// partial in order, then the eight in order.  The first nw values ([9][Ci][Co]) go to gw ([9][Co][Ci]), the
// others to gb.
__global__ void __launch_bounds__(256) k_sum_parts(const float4* part, int S, int n4, int nw4, int Ci, int Co, float* gw,
                                                   float* gb)
{
    __shared__ float4 red[8][32];
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    pdl_wait();
    pdl_trigger();
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < n4) {
#pragma unroll 4
        for (int s = k; s < S; s += 8) {
            const float4 q = part[(long long)s * n4 + i];
            v.x += q.x;
            v.y += q.y;
            v.z += q.z;
            v.w += q.w;
        }
    }
    red[k][lane] = v;
    __syncthreads();
    if (k != 0 || i >= n4) return;
#pragma unroll
    for (int q = 1; q < 8; ++q) {
        const float4 w = red[q][lane];
        v.x += w.x;
        v.y += w.y;
        v.z += w.z;
        v.w += w.w;
    }
    float* o = gb + 4LL * (i - nw4);
    long long step = 1;
    if (i < nw4) {
        const int r = 4 * i / Co, co = 4 * i - r * Co, t = r / Ci, ci = r - t * Ci;
        o = gw + ((long long)t * Co + co) * Ci + ci;
        step = Ci;
    }
    o[0] = v.x;
    o[step] = v.y;
    o[2 * step] = v.z;
    o[3 * step] = v.w;
}

// ------------------------------------------------------------------ weights

// 16-byte units of the packed layouts: unit u of a layer's forward form is (chunk, tap, half, co), of
// its data-gradient form (chunk over o, tap, half, c)
__global__ void k_conv_pack(const __grid_constant__ PackArgs p)
{
    pdl_trigger();               // a convolution of w_late reads nothing of this before it has waited
    const PackLayer L = p.L[blockIdx.y];
    const int cof = (L.Co + 15) / 16 * 16, cid = (L.Ci + 15) / 16 * 16;
    const int nf = L.fwd ? L.Ci / 16 * 18 * cof : 0, nd = L.dgrad ? L.Co / 16 * 18 * cid : 0;
    const int nt = L.wt ? 9 * L.Co * L.Ci : 0;
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < nf + nd + nt; u += gridDim.x * blockDim.x) {
        if (u < nf) {
            const int co = u % cof, r = u / cof, h = r & 1, t = (r >> 1) % 9, k = (r >> 1) / 9;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (co < L.Co) v = *reinterpret_cast<const uint4*>(L.w + ((long long)t * L.Co + co) * L.Ci + 16 * k + 8 * h);
            reinterpret_cast<uint4*>(L.fwd)[u] = v;
        } else if (u < nf + nd) {
            const int q = u - nf;
            const int c = q % cid, r = q / cid, h = r & 1, t = (r >> 1) % 9, k = (r >> 1) / 9;
            __align__(16) bf16 v[8];
            for (int e = 0; e < 8; ++e)
                v[e] = c < L.Ci ? L.w[((long long)(8 - t) * L.Co + 16 * k + 8 * h + e) * L.Ci + c] : __float2bfloat16_rn(0.f);
            reinterpret_cast<uint4*>(L.dgrad)[q] = *reinterpret_cast<const uint4*>(v);
        } else {
            const int q = u - nf - nd;               // wt[t'][c][o] = w[8 - t'][o][c]
            const int o = q % L.Co, r = q / L.Co, c = r % L.Ci, t = r / L.Ci;
            L.wt[q] = L.w[((long long)(8 - t) * L.Co + o) * L.Ci + c];
        }
    }
}

// SMs of the current device
int sm_count()
{
    static std::atomic<int> known[64];
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 152;
    if (dev < 64 && (n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 152;
    if (dev < 64) known[dev].store(n, std::memory_order_relaxed);
    return n;
}

int* g_conv_err = nullptr;      // device flag: a tcgen05 kernel's bounded wait gave up

cudaError_t conv_err_init()
{
    if (g_conv_err) return cudaSuccess;
    cudaError_t e = cudaMalloc(&g_conv_err, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(g_conv_err, 0, sizeof(int));
    return e;
}

template <int MT, bool DIRECT>
cudaError_t launch_tc(const ConvArgs& a, const ConvGeo& g, unsigned m_tiles, int n_cot, cudaStream_t s, bool pdl)
{
    static unsigned long long attr = 0;      // per device
    if (!done_on_device(attr)) {
        cudaError_t e = cudaFuncSetAttribute(k_conv_tc<MT, DIRECT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) {
            attr = 0;
            return e;
        }
    }
    const size_t smem = TC_HEAD + (size_t)g.npix * 4 + (size_t)g.slots * g.cw * (g.npix * 32 + 288 * g.cop);
    return launch_pdl(k_conv_tc<MT, DIRECT>, dim3(m_tiles, n_cot), TC_THREADS, smem, s, pdl, a, g, g_conv_err);
}

}  // namespace

int* conv_err_flag() { return g_conv_err; }

cudaError_t conv_pack(const PackArgs& p, cudaStream_t s)
{
    // a unit per thread for a single layer; the network's layers together fill the GPU with 48 CTAs each
    long long blocks = 48;
    if (p.n == 1) {
        const PackLayer& L = p.L[0];
        const long long u = (L.fwd ? conv_pack_elems(L.Ci, L.Co) / 8 : 0) + (L.dgrad ? conv_pack_elems(L.Co, L.Ci) / 8 : 0) +
                            (L.wt ? 9LL * L.Ci * L.Co : 0);
        blocks = std::max(1LL, std::min((u + 255) / 256, 8LL * sm_count()));
    }
    k_conv_pack<<<dim3((unsigned)blocks, p.n), 256, 0, s>>>(p);
    return cudaGetLastError();
}

// How a call's positions and channels are split over CTAs.
struct ConvSplit {
    bool flat;
    int mt, cop, n_cot;      // MMA tiles and channels per CTA, CTAs of the channels
    long long tiles;         // CTAs of the positions
    long long ctas() const { return tiles * n_cot; }
};

static ConvSplit conv_split(int B, int H, int W, int Co)
{
    const int n_sm = sm_count(), cpk = (Co + 15) / 16 * 16;
    const long long flat_n = (long long)B * (H + 1) * (W + 1);
    ConvSplit c;
    c.flat = W <= 128 && flat_n < (1LL << 30);
    auto tiles = [&](int mt) -> long long {
        if (c.flat) return (flat_n + 128 * mt - 1) / (128 * mt);
        return (long long)((W + 29) / 30) * ((H + 4 * mt - 1) / (4 * mt)) * B;
    };
    // channels per CTA: all up to 128, in equal parts beyond; MMA tiles per CTA: as many as leave one and
    // a half CTAs per SM, fit half the tensor memory and (tiles form, 4 rows each) hold rows of the image
    // (1 x 100000, 16 -> 16 channels: 79 us with four of them, 60 with one); then, where the CTAs would leave
    // SMs empty, the channels are split further (each part stages the input again)
    c.n_cot = (cpk + 127) / 128;
    c.cop = ((cpk + c.n_cot - 1) / c.n_cot + 15) / 16 * 16;
    c.mt = 4;
    while (c.mt > 1 && (c.mt * c.cop > 256 || 2 * tiles(c.mt) * c.n_cot < 3 * n_sm || (!c.flat && H <= 2 * c.mt))) c.mt /= 2;
    while (c.cop > 16 && 4 * tiles(c.mt) * ((cpk + c.cop - 1) / c.cop) < 3 * n_sm) c.cop = (c.cop / 2 + 15) / 16 * 16;
    c.n_cot = (cpk + c.cop - 1) / c.cop;
    c.tiles = tiles(c.mt);
    return c;
}

bool conv_direct(int B, int H, int W, int Ci, int Co)
{
    const ConvSplit c = conv_split(B, H, W, Co);
    const int n_sm = sm_count();
    return 2 * c.ctas() <= 3 * n_sm || (Ci * (long long)c.cop <= 1024 && (c.ctas() <= 3 * n_sm || c.mt == 1));
}

cudaError_t conv_tc(const ConvArgs& a, cudaStream_t s, bool pdl)
{
    if (a.Ci % 16 != 0 || (!a.wp && !a.w) || !conv_tc_fits(a.B, a.H, a.W)) return cudaErrorInvalidValue;
    const cudaError_t e = conv_err_init();
    if (e != cudaSuccess) return e;
    const ConvSplit c = conv_split(a.B, a.H, a.W, a.Co);
    const int mt = c.mt, n_cot = c.n_cot;
    ConvGeo g = {};
    g.cpk = (a.Co + 15) / 16 * 16;
    g.cop = c.cop;
    g.flat = c.flat ? 1 : 0;
    g.pitch = g.flat ? a.W + 1 : 32;
    g.tx = (a.W + 29) / 30;
    g.ty = (a.H + 4 * mt - 1) / (4 * mt);
    // positions: a multiple of 4 that is not one of 8, which spreads the k-halves over the banks
    g.npix = g.flat ? 128 * mt + 2 * g.pitch + 2 : (4 * mt + 2) * 32 + 8;
    g.npix = (g.npix + 3) / 8 * 8 + 4;
    g.d0 = FastDiv((unsigned)(g.flat ? g.pitch : g.tx));
    g.d1 = FastDiv((unsigned)(g.flat ? a.H + 1 : g.tx * g.ty));
    g.ncol = 32;
    while ((int)g.ncol < mt * g.cop) g.ncol *= 2;
    // stages: all chunks where one CTA has an SM to itself, else what lets two share it; the widest
    // stage of which two fit
    const int cbytes = g.npix * 32 + 288 * g.cop, nchunk = a.Ci / 16;
    const int room = (c.ctas() <= sm_count() ? 220 : 110) * 1024 - TC_HEAD - g.npix * 4;
    for (g.cw = 4, g.lgh = 3; g.cw > 1; g.cw /= 2, --g.lgh)
        if (nchunk % g.cw == 0 && std::min(2, nchunk / g.cw) * g.cw * cbytes <= room) break;
    g.slots = std::max(1, std::min(std::min(nchunk / g.cw, TC_SLOTS), room / (g.cw * cbytes)));
    if (c.tiles > 0x7fffffffLL || n_cot > 65535) return cudaErrorInvalidConfiguration;
    const unsigned m = (unsigned)c.tiles;
    switch (2 * mt + (a.wp ? 0 : 1)) {
    case 9: return launch_tc<4, true>(a, g, m, n_cot, s, pdl);
    case 8: return launch_tc<4, false>(a, g, m, n_cot, s, pdl);
    case 5: return launch_tc<2, true>(a, g, m, n_cot, s, pdl);
    case 4: return launch_tc<2, false>(a, g, m, n_cot, s, pdl);
    case 3: return launch_tc<1, true>(a, g, m, n_cot, s, pdl);
    default: return launch_tc<1, false>(a, g, m, n_cot, s, pdl);
    }
}

cudaError_t conv_mma(const ConvArgs& a, cudaStream_t s)
{
    dim3 grid((a.W + CT_W - 1) / CT_W, (a.H + CT_H - 1) / CT_H, a.B * ((a.Co + CT_CO - 1) / CT_CO));
    const long long ctas = (long long)grid.x * grid.y * grid.z, n_sm = sm_count();
    if (!a.yf && (a.ldy % 2 != 0 || ((uintptr_t)(a.y + a.yoff) & 3) != 0)) k_conv3x3<4, true><<<grid, 128, 0, s>>>(a);
    else if ((ctas + 5 * n_sm - 1) / (5 * n_sm) < (ctas + 4 * n_sm - 1) / (4 * n_sm)) k_conv3x3<5, false><<<grid, 128, 0, s>>>(a);
    else k_conv3x3<4, false><<<grid, 128, 0, s>>>(a);
    return cudaGetLastError();
}

// Units and partial sums of a layer's weight gradient; room: floats of the partial sums' buffer (0: as
// many as wanted).  Returns S.
static int wgrad_geo(int B, int H, int W, int Ci, int Co, long long room, WgradGeo& g)
{
    const int n_sm = sm_count();
    const int nb_o = (Co + WG_NMAX - 1) / WG_NMAX, nb_i = (Ci + 127) / 128;
    g.cob = ((Co + nb_o - 1) / nb_o + 15) / 16 * 16;
    g.cib = ((Ci / 8 + nb_i - 1) / nb_i) * 8;
    g.ncol = 32;
    while ((int)g.ncol < 9 * g.cob) g.ncol *= 2;
    g.n = 9LL * Ci * Co + Co;
    g.strips = (W + 31) / 32;
    // one CTA per SM (two where the accumulators leave half the tensor memory), each with several units
    // so that the last ones do not leave SMs idle; shorter units where the image is small
    const int occ = (int)(512 / g.ncol);
    long long S = std::max(1, occ * n_sm / (nb_o * nb_i));
    if (room > 0) S = std::max(1LL, std::min(S, room / g.n));
    for (g.RB = 32;; g.RB /= 2) {
        g.rbs = (H + g.RB - 1) / g.RB;
        if ((long long)B * g.strips * g.rbs >= 5 * S || g.RB == 2) break;
    }
    const long long units = (long long)B * g.strips * g.rbs;
    g.units = (int)std::min<long long>(units, 0x7fffffff);
    S = std::min(S, units);
    const int sbytes = (g.cib / 8 + 3 * (g.cob / 8)) * WG_P * 16;
    const int bytes = (occ > 1 ? 108 : 216) * 1024 - TC_HEAD - 17 * WG_P * 16;
    g.slots = std::max(4, std::min(TC_SLOTS, bytes / sbytes));
    return (int)S;
}

long long wgrad_part_elems(int B, int H, int W, int Ci, int Co)
{
    WgradGeo g;
    return wgrad_geo(B, H, W, Ci, Co, 0, g) * g.n;
}

cudaError_t conv_wgrad(cudaStream_t s, const bf16* x, long long ldx, int xoff, const bf16* gz, int B, int H, int W,
                       int Ci, int Co, float* part, long long room, float* gw, float* gb, bool pdl)
{
    cudaError_t e = conv_err_init();
    if (e != cudaSuccess) return e;
    static unsigned long long attr = 0;      // per device
    if (!done_on_device(attr)) {
        e = cudaFuncSetAttribute(k_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) {
            attr = 0;
            return e;
        }
    }
    WgradGeo g;
    const int S = wgrad_geo(B, H, W, Ci, Co, room, g);
    WgradArgs a = {};
    a.x = x; a.ldx = ldx; a.xoff = xoff; a.gz = gz; a.part = part;
    a.B = B; a.H = H; a.W = W; a.Ci = Ci; a.Co = Co;
    // the last stage's operand of 128 channels may reach past its own channels: 16 groups of slack
    const size_t smem = TC_HEAD + (size_t)g.slots * (g.cib / 8 + 3 * (g.cob / 8)) * WG_P * 16 + 17 * WG_P * 16;
    e = launch_pdl(k_wgrad_tc, dim3(S, (Ci + g.cib - 1) / g.cib, (Co + g.cob - 1) / g.cob), TC_THREADS, smem, s, pdl, a, g,
                   g_conv_err);
    if (e != cudaSuccess) return e;
    const int n4 = (int)(g.n / 4), nw4 = (int)(9LL * Ci * Co / 4);
    return launch_pdl(k_sum_parts, dim3((n4 + 31) / 32), 256, 0, s, true, reinterpret_cast<const float4*>(part), S, n4, nw4,
                      Ci, Co, gw, gb);
}

}  // namespace net
}  // namespace vlb
