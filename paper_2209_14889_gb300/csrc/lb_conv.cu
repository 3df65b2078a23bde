// lb_conv.cu -- 3x3 convolutions on NHWC BF16 activations with FP32 accumulation (the network of
// the learned stepper): forward passes and data gradients, as implicit GEMMs with the pixels as M,
// the output channels as N and K = 9 Ci.
#include <algorithm>

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
__device__ __forceinline__ void ldsm_x4_t(unsigned (&r)[4], const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
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

__global__ void __launch_bounds__(128) k_conv3x3(const ConvArgs a)
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
                    *reinterpret_cast<__nv_bfloat162*>(a.y + o) = __floats2bfloat162_rn(v0, v1);
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
// swizzle: input [2 k-halves][positions][8], weights [9 taps][2 k-halves][cop][8]; 8-row groups 128
// bytes apart.
//
// Four warps copy the input (cp.async, the position's address formed once for all chunks), one warp
// the weights (bulk copies of the packed layout, conv_pack), one thread issues the MMAs; the chunks
// go through up to 16 stages, each with a barrier for its input, its weights and its release by the
// MMAs that read it (tcgen05.commit).  The four copying warps then store the result.
//
// What bounds it: at 32 channels the 128 x 16 input operand of every MMA is read from shared memory
// (4 KB, 32 cycles) for half as many cycles of tensor work; at few CTAs (the 1/4 and 1/8 resolution
// layers) the latency of one CTA's chain, which is why all chunks' copies are issued ahead and the
// channels are split until every SM has a CTA.

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
    for (long it = 0; it < (1L << 22) && !done; ++it) {
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
__device__ __forceinline__ void tc_mma(unsigned d, uint64_t ad, uint64_t bd, uint32_t idesc, int acc)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void tc_ld16(unsigned (&v)[16], unsigned taddr)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
        "%13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

constexpr int TC_THREADS = 192;                  // 4 copying and storing warps, MMA warp, weights warp
constexpr int TC_SLOTS = 16;                     // most stages
constexpr int TC_HEAD = 512;                     // shared bytes of the barriers

struct ConvGeo {
    int flat, pitch, npix;                       // npix: staged positions
    int cop, slots, tx, ty;                      // channels per CTA, stages, tile grid (tiles form)
    int cpk;                                     // channels of the packed weights
    unsigned ncol;                               // tensor-memory columns (a power of two >= 32)
};

// shared state of a tcgen05 kernel ahead of its stages
struct TcShared {
    uint64_t xfull[TC_SLOTS], wfull[TC_SLOTS], empty[TC_SLOTS], done;
    unsigned tmem;
    int fail;
};
static_assert(sizeof(TcShared) <= TC_HEAD, "barriers fit ahead of the stages");

// output position -> pixel (b, y, x); false where there is none
template <int MT>
__device__ __forceinline__ bool out_pixel(const ConvArgs& a, const ConvGeo& g, int mt, int m, int& b, int& y, int& x)
{
    if (g.flat) {
        const int Q = (int)blockIdx.x * (128 * MT) + 128 * mt + m;
        const int row = Q / g.pitch;
        x = Q - row * g.pitch;
        b = row / (a.H + 1);
        y = row - b * (a.H + 1);
        return x < a.W && y < a.H && b < a.B;
    }
    const int per = g.tx * g.ty;
    b = (int)blockIdx.x / per;
    const int r = (int)blockIdx.x - b * per;
    const int c = m & 31;
    y = (r / g.tx) * (4 * MT) + 4 * mt + (m >> 5);
    x = (r % g.tx) * 30 + c;
    return c < 30 && x < a.W && y < a.H;
}

// element offset of the pixel at staged position p (without the channel), or -1 where it is padding
template <int MT>
__device__ __forceinline__ long long in_pixel(const ConvArgs& a, const ConvGeo& g, int p)
{
    int b, y, x;
    if (g.flat) {
        const int Q = (int)blockIdx.x * (128 * MT) - g.pitch - 1 + p;
        if (Q < 0) return -1;
        const int row = Q / g.pitch;
        x = Q - row * g.pitch;
        b = row / (a.H + 1);
        y = row - b * (a.H + 1);
        if (b >= a.B) return -1;
    } else {
        const int per = g.tx * g.ty;
        b = (int)blockIdx.x / per;
        const int r = (int)blockIdx.x - b * per;
        y = (r / g.tx) * (4 * MT) - 1 + (p >> 5);
        x = (r % g.tx) * 30 - 1 + (p & 31);
        if (p >= (4 * MT + 2) * 32 || y < 0 || x < 0) return -1;
    }
    if (x >= a.W || y >= a.H) return -1;
    return (((long long)b * a.H + y) * a.W + x) * a.ldx + a.xoff;
}

template <int MT>
__global__ void __launch_bounds__(TC_THREADS) k_conv_tc(const __grid_constant__ ConvArgs a, const __grid_constant__ ConvGeo g,
                                                        int* err)
{
    // copies per thread and chunk: 2 npix / 128, npix <= max(128 MT + 72, 128 MT + 260)
    constexpr int NU = (2 * (128 * MT + 260) + 127) / 128;
    extern __shared__ __align__(128) unsigned char smem[];
    TcShared& S = *reinterpret_cast<TcShared*>(smem);
    const int xbytes = g.npix * 32, wbytes = 288 * g.cop, sbytes = xbytes + wbytes;
    const unsigned stage0 = smem_u32(smem) + TC_HEAD;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int co0 = blockIdx.y * g.cop;
    const int nchunk = a.Ci / 16, slots = g.slots;

    if (tid == 0) {
        for (int s = 0; s < slots; ++s) {
            mbar_init(&S.xfull[s], 128);
            mbar_init(&S.wfull[s], 1);
            mbar_init(&S.empty[s], 1);
        }
        mbar_init(&S.done, 1);
        S.fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem)),
                     "r"(g.ncol));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = S.tmem;

    bool ok = true;
    if (warp < 4) {
        // ---- input: 16-byte units (position, k-half); a thread's units and their addresses are the
        // same in every chunk, 32 bytes further on
        long long src[NU];
#pragma unroll
        for (int i = 0; i < NU; ++i) {
            const int u = tid + 128 * i;
            src[i] = u < 2 * g.npix ? in_pixel<MT>(a, g, u >> 1) : -1;
        }
        pdl_wait();                       // the input is the result of the kernel before this one
        for (int k = 0; k < nchunk && ok; ++k) {
            const int s = k % slots;
            if (k >= slots) ok = mbar_wait(&S.empty[s], (unsigned)((k / slots - 1) & 1));
            if (!ok) break;
            const unsigned dst = stage0 + (unsigned)(s * sbytes);
            const bf16* base = a.x + 16 * k + 8 * (tid & 1);
            const int h = tid & 1;
#pragma unroll
            for (int i = 0; i < NU; ++i) {
                const int u = tid + 128 * i;
                if (u < 2 * g.npix)
                    cp_async16(dst + (unsigned)((h * g.npix + (u >> 1)) * 16), src[i] >= 0 ? base + src[i] : a.x,
                               src[i] >= 0 ? 16 : 0);
            }
            cp_async_arrive(&S.xfull[s]);
        }
        pdl_trigger();
    } else if (warp == 5) {
        // ---- weights: 18 bulk copies (tap, k-half) of the CTA's channels per chunk, one per lane
        const unsigned nb = (unsigned)min(g.cop, g.cpk - co0) * 16u;
        int issued = 0;
        for (int k = 0; k < nchunk && ok; ++k) {
            const int s = k % slots;
            if (k >= slots) ok = __all_sync(0xffffffffu, mbar_wait(&S.empty[s], (unsigned)((k / slots - 1) & 1)));
            if (!ok) break;
            if (lane == 0) mbar_expect_tx(&S.wfull[s], 18u * nb);
            __syncwarp();
            if (lane < 18)
                bulk_copy(stage0 + (unsigned)(s * sbytes + xbytes + lane * g.cop * 16),
                          a.wp + (((long long)k * 18 + lane) * g.cpk + co0) * 8, nb, &S.wfull[s]);
            issued = k + 1;
        }
        // the CTA does not end with a weights copy in flight, whatever happened above
        for (int k = max(0, issued - slots); k < issued; ++k)
            mbar_wait(&S.wfull[k % slots], (unsigned)((k / slots) & 1));
    } else if (lane == 0) {
        // ---- MMAs
        const uint32_t idesc =
            (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(g.cop >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        for (int k = 0; k < nchunk && ok; ++k) {
            const int s = k % slots;
            const unsigned par = (unsigned)((k / slots) & 1);
            ok = mbar_wait(&S.xfull[s], par) && mbar_wait(&S.wfull[s], par);
            if (!ok) break;
            // the input was written through the generic proxy, the tensor core reads through the
            // asynchronous one
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const unsigned sx = stage0 + (unsigned)(s * sbytes), sw = sx + (unsigned)xbytes;
            for (int t = 0; t < 9; ++t) {
                const uint64_t bd = tc_desc(sw + (unsigned)(t * 2 * g.cop * 16), (unsigned)(g.cop * 16), 128);
                const int p0 = (t / 3) * g.pitch + t % 3;
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
                    tc_mma(tmem + (unsigned)(mt * g.cop), tc_desc(sx + (unsigned)((p0 + 128 * mt) * 16), (unsigned)(g.npix * 16), 128),
                           bd, idesc, (k > 0 || t > 0) ? 1 : 0);
            }
            tc_commit(&S.empty[s]);
        }
        if (ok) tc_commit(&S.done);
    }
    if (!ok) S.fail = 1;

    if (warp < 4) {
        if (ok) ok = mbar_wait(&S.done, 0);
        if (!ok) S.fail = 1;
        cp_async_wait_all();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok) {
            // warp w holds the positions 32 w .. of each tile, the columns are the channels co0 ..
            for (int mt = 0; mt < MT; ++mt) {
                int b, y, x;
                const bool valid = out_pixel<MT>(a, g, mt, tid, b, y, x);
                const long long pix = ((long long)b * a.H + y) * a.W + x;
                const long long o0 = pix * a.ldy + a.yoff + co0;
                for (int j = 0; j < g.cop; j += 16) {
                    unsigned v[16];
                    tc_ld16(v, tmem + ((unsigned)(warp * 32) << 16) + (unsigned)(mt * g.cop + j));
                    if (!valid) continue;
                    float f[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int co = co0 + j + e;
                        float val = __uint_as_float(v[e]) + ((a.bias && co < a.Co) ? __ldg(a.bias + co) : 0.f);
                        if (a.act) val = val > 0.f ? val : SLOPE * val;
                        f[e] = val;
                    }
                    const bool whole = co0 + j + 16 <= a.Co;
                    if (a.yf) {
                        if (whole && ((o0 + j) & 3) == 0) {
#pragma unroll
                            for (int e = 0; e < 16; e += 4) {
                                const float4 q = make_float4(f[e], f[e + 1], f[e + 2], f[e + 3]);
                                *reinterpret_cast<float4*>(a.yf + o0 + j + e) = q;
                                if (a.yf2) *reinterpret_cast<float4*>(a.yf2 + o0 + j + e) = q;
                            }
                        } else {
                            for (int e = 0; e < 16; ++e)
                                if (co0 + j + e < a.Co) {
                                    a.yf[o0 + j + e] = f[e];
                                    if (a.yf2) a.yf2[o0 + j + e] = f[e];
                                }
                        }
                        continue;
                    }
                    __nv_bfloat162 r[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) r[e] = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
                    if (a.ym) {                     // the gradient through the layer below's LeakyReLU
                        const uint4* mp = reinterpret_cast<const uint4*>(a.ym + pix * a.ldm + a.moff + co0 + j);
                        const uint4 m4[2] = {__ldg(mp), __ldg(mp + 1)};
                        const __nv_bfloat162* mv = reinterpret_cast<const __nv_bfloat162*>(m4);
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const float2 gg = __bfloat1622float2(r[e]), mm = __bfloat1622float2(mv[e]);
                            r[e] = __floats2bfloat162_rn(mm.x > 0.f ? gg.x : SLOPE * gg.x, mm.y > 0.f ? gg.y : SLOPE * gg.y);
                        }
                    }
                    if (whole && ((o0 + j) & 7) == 0) {
                        const uint4 w0 = *reinterpret_cast<const uint4*>(r), w1 = *reinterpret_cast<const uint4*>(r + 4);
                        *reinterpret_cast<uint4*>(a.y + o0 + j) = w0;
                        *reinterpret_cast<uint4*>(a.y + o0 + j + 8) = w1;
                        if (a.up) {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                bf16* d = a.up + (((long long)b * 2 * a.H + 2 * y + (q >> 1)) * 2 * a.W + 2 * x + (q & 1)) * a.ldu +
                                          co0 + j;
                                *reinterpret_cast<uint4*>(d) = w0;
                                *reinterpret_cast<uint4*>(d + 8) = w1;
                            }
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            if (co0 + j + e < a.Co) a.y[o0 + j + e] = e & 1 ? r[e >> 1].y : r[e >> 1].x;
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (S.fail && tid == 0) atomicExch(err, 1);
    if (warp == 4) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(g.ncol));
    }
}

// ------------------------------------------------------------------ weight gradient

constexpr int WG_CO = 64, WG_CI = 16;           // output block of gw per CTA: [9][64][16]
constexpr int DZS = WG_CO + 8;                  // shared row of 64 channels + 8 pad (144 bytes)

struct WgradArgs {
    const bf16* x;          // layer input (pixel stride ldx, offset xoff)
    long long ldx;
    int xoff;
    const bf16* gz;         // gradient at the layer's pre-activation output [P][Co] (stride ldz)
    long long ldz;
    float* part;            // [S][9][Co][Ci] partial sums
    int B, H, W, Ci, Co, S;
};

__global__ void __launch_bounds__(128) k_conv_wgrad(const WgradArgs a)
{
    __shared__ __align__(16) bf16 sdz[CT_H * CT_W * DZS];
    __shared__ __align__(16) bf16 sx[CT_IH * CT_IW * PS];
    const int co0 = blockIdx.x * WG_CO, ci0 = blockIdx.y * WG_CI, s = blockIdx.z;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tiles_x = (a.W + CT_W - 1) / CT_W, tiles_y = (a.H + CT_H - 1) / CT_H;
    const int n_tiles = a.B * tiles_x * tiles_y;
    float acc[9][2][4];
#pragma unroll
    for (int t = 0; t < 9; ++t)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[t][j][k] = 0.f;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);

    for (int tile = s; tile < n_tiles; tile += a.S) {
        const int b = tile / (tiles_x * tiles_y), r = tile - b * (tiles_x * tiles_y);
        const int ty0 = (r / tiles_x) * CT_H, tx0 = (r % tiles_x) * CT_W;
        // gz tile: 128 pixels x 64 channels (8 chunks of 8)
        for (int q = tid; q < CT_H * CT_W * 8; q += 128) {
            const int p = q >> 3, h = q & 7;
            const int gy = ty0 + p / CT_W, gx = tx0 + p % CT_W;
            uint4 v = zero;
            if (gy < a.H && gx < a.W && co0 + h * 8 < a.Co)
                v = *reinterpret_cast<const uint4*>(a.gz + ((long long)(b * a.H + gy) * a.W + gx) * a.ldz + co0 + h * 8);
            *reinterpret_cast<uint4*>(sdz + p * DZS + h * 8) = v;
        }
        for (int q = tid; q < CT_IH * CT_IW * 2; q += 128) {
            const int p = q >> 1, h = q & 1;
            const int py = p / CT_IW, px = p - py * CT_IW;
            const int gy = ty0 - 1 + py, gx = tx0 - 1 + px;
            uint4 v = zero;
            if (gy >= 0 && gy < a.H && gx >= 0 && gx < a.W)
                v = *reinterpret_cast<const uint4*>(a.x + ((long long)(b * a.H + gy) * a.W + gx) * a.ldx + a.xoff + ci0 +
                                                    h * 8);
            *reinterpret_cast<uint4*>(sx + p * PS + h * 8) = v;
        }
        __syncthreads();
        const int j = lane >> 3, rr = lane & 7;
#pragma unroll 1
        for (int ks = 0; ks < CT_H; ++ks) {             // 16 pixels (one tile row) per k-step
            unsigned A[4];                               // (co, p): rows p of sdz, transposed
            ldsm_x4_t(A, sdz + (ks * CT_W + rr + (j >> 1) * 8) * DZS + warp * 16 + (j & 1) * 8);
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const int dy = t / 3 - 1, dx = t % 3 - 1;
                unsigned Bf[4];                          // (p, ci): rows p of the shifted input
                const int k = rr + (j & 1) * 8;
                ldsm_x4_t(Bf, sx + ((ks + 1 + dy) * CT_IW + (k + 1 + dx)) * PS + (j >> 1) * 8);
                mma_bf16(acc[t][0], A, Bf[0], Bf[1]);
                mma_bf16(acc[t][1], A, Bf[2], Bf[3]);
            }
        }
        __syncthreads();
    }
    const int g = lane >> 2, tq = lane & 3;
#pragma unroll
    for (int t = 0; t < 9; ++t)
#pragma unroll
        for (int jn = 0; jn < 2; ++jn)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const int co = co0 + warp * 16 + g + 8 * hh;
                const int ci = ci0 + jn * 8 + 2 * tq;
                if (co < a.Co) {
                    float* o = a.part + (((long long)s * 9 + t) * a.Co + co) * a.Ci + ci;
                    o[0] = acc[t][jn][2 * hh];
                    o[1] = acc[t][jn][2 * hh + 1];
                }
            }
}

// sum of S partial arrays of n floats, in order: out[i] = sum_s part[s][i]
__global__ void k_sum_parts(const float* part, int S, long long n, float* out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float v = 0.f;
    for (int s = 0; s < S; ++s) v += part[(long long)s * n + i];
    out[i] = v;
}

// bias gradient partials: part[s][o] = sum over pixels p = s, s + S, ... of gz[p][o]
__global__ void k_bias_parts(const bf16* gz, long long ldz, long long P, int Co, int S, float* part)
{
    const int o = blockIdx.x * blockDim.x + threadIdx.x, s = blockIdx.y;
    if (o >= Co) return;
    float v = 0.f;
    for (long long p = s; p < P; p += S) v += __bfloat162float(gz[p * ldz + o]);
    part[(long long)s * Co + o] = v;
}

// ------------------------------------------------------------------ weights

// 16-byte units of the packed layouts: unit u of a layer's forward form is (chunk, tap, half, co), of
// its data-gradient form (chunk over o, tap, half, c)
__global__ void k_conv_pack(const __grid_constant__ PackArgs p)
{
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

int sm_count()
{
    int dev = 0, n = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
}

int* g_conv_err = nullptr;      // device flag: a tcgen05 kernel's bounded wait gave up

template <int MT>
cudaError_t launch_tc(const ConvArgs& a, const ConvGeo& g, unsigned m_tiles, int n_cot, cudaStream_t s, bool pdl)
{
    static unsigned long long attr = 0;      // per device
    if (!done_on_device(attr)) {
        cudaError_t e = cudaFuncSetAttribute(k_conv_tc<MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) {
            attr = 0;
            return e;
        }
    }
    const size_t smem = TC_HEAD + (size_t)g.slots * (g.npix * 32 + 288 * g.cop);
    return launch_pdl(k_conv_tc<MT>, dim3(m_tiles, n_cot), TC_THREADS, smem, s, pdl, a, g, g_conv_err);
}

}  // namespace

int* conv_err_flag() { return g_conv_err; }

cudaError_t conv_pack(const PackArgs& p, cudaStream_t s)
{
    k_conv_pack<<<dim3(48, p.n), 256, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t conv_tc(const ConvArgs& a, cudaStream_t s, bool pdl)
{
    if (a.Ci % 16 != 0) return cudaErrorInvalidValue;
    if (!g_conv_err) {
        cudaError_t e = cudaMalloc(&g_conv_err, sizeof(int));
        if (e == cudaSuccess) e = cudaMemset(g_conv_err, 0, sizeof(int));
        if (e != cudaSuccess) return e;
    }
    static const int n_sm = sm_count();
    ConvGeo g = {};
    g.cpk = (a.Co + 15) / 16 * 16;
    const long long flat_n = (long long)a.B * (a.H + 1) * (a.W + 1);
    g.flat = a.W <= 128 && flat_n < (1LL << 30) ? 1 : 0;
    g.pitch = g.flat ? a.W + 1 : 32;
    g.tx = (a.W + 29) / 30;
    auto tiles = [&](int mt) -> long long {
        if (g.flat) return (flat_n + 128 * mt - 1) / (128 * mt);
        return (long long)g.tx * ((a.H + 4 * mt - 1) / (4 * mt)) * a.B;
    };
    // channels per CTA: all up to 128, in equal parts beyond; MMA tiles per CTA: as many as leave two
    // CTAs per SM and fit half the tensor memory; then, where the CTAs would leave SMs empty, the
    // channels are split further (each part stages the input again)
    int n_cot = (g.cpk + 127) / 128;
    g.cop = ((g.cpk + n_cot - 1) / n_cot + 15) / 16 * 16;
    int mt = 4;
    while (mt > 1 && (mt * g.cop > 256 || tiles(mt) * n_cot < 2 * n_sm)) mt /= 2;
    while (g.cop > 16 && tiles(mt) * ((g.cpk + g.cop - 1) / g.cop) < n_sm) g.cop = (g.cop / 2 + 15) / 16 * 16;
    n_cot = (g.cpk + g.cop - 1) / g.cop;
    g.ty = (a.H + 4 * mt - 1) / (4 * mt);
    g.npix = g.flat ? 128 * mt + 2 * g.pitch + 2 : (4 * mt + 2) * 32 + 8;
    g.ncol = 32;
    while ((int)g.ncol < mt * g.cop) g.ncol *= 2;
    // stages: all chunks where one CTA has an SM to itself, else what lets two share it
    const int sbytes = g.npix * 32 + 288 * g.cop;
    const int room = tiles(mt) * n_cot <= n_sm ? 220 * 1024 : 110 * 1024;
    g.slots = std::max(1, std::min(std::min(a.Ci / 16, TC_SLOTS), (room - TC_HEAD) / sbytes));
    const long long m_tiles = tiles(mt);
    if (m_tiles > 0x7fffffffLL || n_cot > 65535) return cudaErrorInvalidConfiguration;
    switch (mt) {
    case 4: return launch_tc<4>(a, g, (unsigned)m_tiles, n_cot, s, pdl);
    case 2: return launch_tc<2>(a, g, (unsigned)m_tiles, n_cot, s, pdl);
    default: return launch_tc<1>(a, g, (unsigned)m_tiles, n_cot, s, pdl);
    }
}

cudaError_t conv_mma(const ConvArgs& a, cudaStream_t s)
{
    dim3 grid((a.W + CT_W - 1) / CT_W, (a.H + CT_H - 1) / CT_H, a.B * ((a.Co + CT_CO - 1) / CT_CO));
    k_conv3x3<<<grid, 128, 0, s>>>(a);
    return cudaGetLastError();
}

int wgrad_splits(int B, int H, int W)
{
    const int tiles = B * ((W + CT_W - 1) / CT_W) * ((H + CT_H - 1) / CT_H);
    return tiles < 64 ? tiles : 64;
}

long long wgrad_part_elems(int B, int H, int W, int Ci, int Co)
{
    return (long long)wgrad_splits(B, H, W) * std::max<long long>(9LL * Ci * Co, Co);
}

cudaError_t conv_wgrad(cudaStream_t s, const bf16* x, long long ldx, int xoff, const bf16* gz, int B, int H, int W,
                       int Ci, int Co, float* part, float* gw, float* gb)
{
    const int S = wgrad_splits(B, H, W);
    WgradArgs a;
    a.x = x; a.ldx = ldx; a.xoff = xoff; a.gz = gz; a.ldz = Co; a.part = part;
    a.B = B; a.H = H; a.W = W; a.Ci = Ci; a.Co = Co; a.S = S;
    dim3 grid((Co + WG_CO - 1) / WG_CO, Ci / WG_CI, S);
    k_conv_wgrad<<<grid, 128, 0, s>>>(a);
    const long long nw = 9LL * Co * Ci;
    k_sum_parts<<<(unsigned)((nw + 255) / 256), 256, 0, s>>>(part, S, nw, gw);
    const long long P = (long long)B * H * W;
    k_bias_parts<<<dim3((Co + 127) / 128, S), 128, 0, s>>>(gz, Co, P, Co, S, part);
    k_sum_parts<<<(unsigned)((Co + 255) / 256), 256, 0, s>>>(part, S, Co, gb);
    return cudaGetLastError();
}

}  // namespace net
}  // namespace vlb
