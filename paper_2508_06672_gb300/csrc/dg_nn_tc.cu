// dg_nn_tc.cu -- the proposal network's 3 x 3 convolutions on the tensor
// cores (tcgen05, sm_103a): BF16 activations and weights, FP32 accumulation.
//
// Both are implicit GEMMs with the accumulator in tensor memory and the
// operands in shared memory (no swizzle, K-major canonical layout: 8-row x
// 16-byte core matrices):
//
//   forward / data gradient: rows = 128 consecutive pixels of one image
//     row (two image rows per CTA, one accumulator each), columns = output
//     channels, K = (input channel, tap) pairs:
//       y[n,o,i,j] = b[o] + sum_{c,u,v} w[o,c,u,v] x[n,c,i+u-1,j+v-1]
//     The data gradient is the same product with dy as the input, the
//     weights transposed (input and output channels swapped) and the taps
//     flipped:
//       dx[n,c,i,j] = sum_{o,u,v} w[o,c,u,v] dy[n,o,i-u+1,j-v+1]
//     The input rows a CTA needs are staged once per block of 32 channels;
//     each tap's A operand is that staging seen through a shifted
//     descriptor (k_conv3x3_tc). The weights are converted to BF16 blocks
//     once per call and stream in by bulk copy.
//   weight gradient: rows = output channels, columns = input channels, one
//     accumulator per tap, K = pixels:
//       dw[o,c,u,v] = sum_{n,i,j} dy[n,o,i,j] x[n,c,i+u-1,j+v-1]
//       db[o]       = sum_{n,i,j} dy[n,o,i,j]   (of the rounded dy, CUDA cores)
//     split over image rows; the partial sums are added in a fixed order. The
//     operands are read MN-major from the same staging of 8-channel pixels
//     (k_conv3x3_dw_tc).
// The FP32 kernels in dg_nn.cu stay as the reference.
#include <cuda_bf16.h>

#include <algorithm>

#include "dg_internal.cuh"

namespace dg {
namespace {

constexpr int kRowsTc = 128;                 // MMA M
constexpr uint32_t kNnWaitLimit = 1u << 24;  // polls before an mbarrier wait gives up

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// byte offset of element (row, k) in a K-major block of 32 K elements
__device__ __forceinline__ uint32_t kmaj(int row, int k)
{
    return (uint32_t)(((row >> 3) * 4 + (k >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// shared-memory descriptor: start >> 4, leading byte offset 128 (K-adjacent
// core matrices), stride byte offset 512 (8-row groups), version 1, no swizzle
__device__ __forceinline__ uint64_t nn_sdesc(uint32_t saddr)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(512 >> 4) << 32) |
           (1ull << 46);
}

// instruction descriptor, kind::f16: FP32 D, BF16 A and B, both K-major,
// N >> 3 at [17, 23), M >> 4 at [24, 29)
__device__ __forceinline__ uint32_t nn_idesc(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kRowsTc >> 4) << 24);
}

__device__ __forceinline__ void nn_mma(uint32_t d, uint64_t ad, uint64_t bd, uint32_t id, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
        "l"(ad), "l"(bd), "r"(id), "r"(acc)
        : "memory");
}

// One lane of a converged warp. The issuing warp runs its loop with all lanes and
// only the instruction itself is predicated: descriptors then stay in uniform
// registers, where a branch on one lane moves each of them there first.
__device__ __forceinline__ uint32_t nn_elect()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(p));
    return p;
}

__device__ __forceinline__ void nn_mma_if(uint32_t lead, uint32_t d, uint64_t ad, uint64_t bd, uint32_t id, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
        "l"(ad), "l"(bd), "r"(id), "r"(acc), "r"(lead)
        : "memory");
}

__device__ __forceinline__ void nn_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void nn_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void nn_mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// bounded wait on an mbarrier phase: false after 2 s of the global timer
// (checked every 256 polls) or kNnWaitLimit polls
__device__ __forceinline__ bool nn_wait(uint32_t bar, uint32_t parity)
{
    uint64_t t0 = 0;
    for (uint32_t i = 0; i < kNnWaitLimit; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((i & 255) == 255) {
            uint64_t now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (t0 == 0) t0 = now;
            else if (now - t0 > 2000000000ull) return false;
        }
    }
    return false;
}

__device__ __forceinline__ void nn_tmem_alloc(uint32_t slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void nn_tmem_free(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void nn_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void nn_fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void nn_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void nn_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

__device__ __forceinline__ uint16_t bf16_bits(float v)
{
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    return *reinterpret_cast<const uint16_t *>(&h);
}

// two values rounded as bf16_bits, the first in the low half
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// Tensor-memory columns of an accumulator of n columns (a power of two >= 32).
__host__ __device__ constexpr int tmem_cols(int n) { return n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : n <= 256 ? 256 : 512; }

}  // namespace

// ---------------------------------------------------------------------------
// Forward and data gradient: halo-staged implicit GEMM. A CTA computes
// kHaloRows output rows x 128 pixels (j0 .. j0 + 127) of image n for output
// channels o0 .. o0 + NT - 1 (NT a multiple of 16, <= 128). K runs over
// (channel block of 32, tap): for each channel block the CTA stages the
// kHaloRows + 2 input rows it needs, pixels j0 - 1 .. j0 + 128, as BF16 in
// shared memory, one 16-byte row per (input row, 8 channels, pixel). In the
// canonical K-major layout a core matrix is then 8 consecutive pixels of one
// 8-channel group, the 8-pixel groups 128 B apart and the channel groups
// kHaloQ * 16 B apart, so the A operand of tap (u, v) for output row r is the
// same staging seen from input row r + u and shifted by v pixels: a
// different descriptor start, nothing gathered per tap. The weights come
// pre-converted (k_conv_tc_wimg: one 32-channel x NT block per (channel
// block, tap) in the canonical layout) by bulk copy, once per CTA where they
// fit beside the staged rows, else through a ring of slots.
//
// One CTA per SM walks the tiles; its warps have a role each and meet only on
// mbarriers: 13 stage input rows into a ring of buffers, one copies weights, one
// issues the MMAs (with all lanes, see nn_elect), eight write finished tiles out
// of one of two accumulator sets while the next tile's products run. (A CTA per
// tile in which every thread staged, one also issued, and all met twice per
// channel block: 222 us for 128 -> 64 channels at 16 x 128 x 128, MMA pipes 8 %
// busy; now 69 us, bound by the staging's loads.) Each output's products are added in the order (channel block, tap,
// K-step).
// x: [B][CI][H][W]; y: [B][CO][H][W]; b may be NULL.
// ---------------------------------------------------------------------------
constexpr int kHaloRows = 2;                                   // output rows per CTA
constexpr int kHaloCB = 32;                                    // input channels per block
constexpr int kHaloQ = kRowsTc + 2;                            // staged pixels per input row
constexpr int kHaloBytes = (kHaloRows + 2) * (kHaloCB / 8) * kHaloQ * 16;
constexpr int kProdWarps = 13;                                 // staging warps: 5 rows of 8 channels a thread
constexpr int kOutWarps = 8;                                   // output warps: four per output row
constexpr int kConvThreads = 32 * (kProdWarps + kOutWarps + 2);  // + weights, MMAs
constexpr int kHaloMax = 4;                                    // staging buffers, at most
constexpr int kWSlots = 64;                                    // weight blocks in shared memory, at most
constexpr int kConvSmem = 224 * 1024;                          // dynamic shared memory, at most

// accumulator columns of one output row (NT rounded up to the 32-column loads)
__host__ __device__ constexpr int acc_stride(int nt) { return (nt + 31) / 32 * 32; }

// elements (16-bit) of the pre-converted weights of a layer with CI inputs and CO outputs
__host__ __device__ inline int64_t wimg_elems(int ci, int co, int nt)
{
    return (int64_t)((co + nt - 1) / nt) * ((ci + kHaloCB - 1) / kHaloCB) * 9 * nt * kHaloCB;
}

// shared-memory descriptor of staged input rows: K-adjacent core matrices
// (8-channel groups) kHaloQ * 16 B apart, 8-pixel groups 128 B apart
__device__ __forceinline__ uint64_t halo_desc(uint32_t saddr)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((kHaloQ * 16) >> 4) << 16) |
           ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}

__device__ __forceinline__ void nn_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void nn_bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Weights of the forward convolution (TR = false: w [CO][CI][3][3]) or of the
// data gradient (TR = true: the forward's w [CI][CO][3][3], transposed, taps
// flipped) as BF16 blocks: block (output block ob, channel block cb, tap) =
// NT output channels x 32 input channels in the canonical K-major layout
// (kmaj), zeros past CO and CI.
template <bool TR>
__device__ __forceinline__ void convert_weights(const float *__restrict__ w, uint16_t *__restrict__ wimg, int CI, int CO, int NT)
{
    const int ncb = (CI + kHaloCB - 1) / kHaloCB, ob = (CO + NT - 1) / NT;
    const int64_t items = (int64_t)ob * ncb * 9 * NT * (kHaloCB / 8);
    for (int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; it < items;
         it += (int64_t)gridDim.x * blockDim.x) {
        const int kg = (int)(it % (kHaloCB / 8));
        const int ol = (int)((it / (kHaloCB / 8)) % NT);
        const int64_t blk = it / ((kHaloCB / 8) * NT);
        const int tap = (int)(blk % 9), cb = (int)((blk / 9) % ncb), obi = (int)(blk / (9 * ncb));
        const int o = obi * NT + ol;
        uint32_t pk[4];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int c = cb * kHaloCB + kg * 8 + e;
            float v = 0.f;
            if (o < CO && c < CI)
                v = TR ? w[((size_t)c * CO + o) * 9 + (8 - tap)] : w[((size_t)o * CI + c) * 9 + tap];
            const uint32_t h = bf16_bits(v);
            pk[e >> 1] = (e & 1) ? (pk[e >> 1] | (h << 16)) : h;
        }
        unsigned char *dst = reinterpret_cast<unsigned char *>(wimg) + (size_t)blk * NT * kHaloCB * 2 + kmaj(ol, kg * 8);
        *reinterpret_cast<uint4 *>(dst) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    }
}

template <bool TR>
__global__ void k_conv_tc_wimg(const float *__restrict__ w, uint16_t *__restrict__ wimg, int CI, int CO, int NT)
{
    convert_weights<TR>(w, wimg, CI, CO, NT);
}

// The forward weights of all layers of a network, layer blockIdx.y: a launch per
// layer takes 4 us for a microsecond of work.
constexpr int kNetLayers = 16;
struct NetWeights {
    const float *w[kNetLayers];
    int64_t off[kNetLayers];  // of the layer's blocks in wimg (elements)
    int CI[kNetLayers], CO[kNetLayers], NT[kNetLayers];
};
// With planes > 0 the last rows of blocks zero the borders of the BF16 tensors: that
// many planes of (H + 2) x (W + 2) 16-byte pixels from act on.
__global__ void k_net_tc_wimg(NetWeights n, uint16_t *__restrict__ wimg, int layers, uint4 *__restrict__ act, int64_t planes,
                              int H, int W)
{
    const int l = blockIdx.y;
    if (l == layers) {
        const int64_t ring = 2 * (int64_t)(W + 2) + 2 * (int64_t)H;
        for (int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; it < planes * ring;
             it += (int64_t)gridDim.x * blockDim.x) {
            const int64_t p = it / ring, r = it % ring;
            const int64_t px = r < W + 2 ? r : r < 2 * (W + 2) ? (int64_t)(H + 1) * (W + 2) + r - (W + 2)
                               : ((r - 2 * (W + 2)) / 2 + 1) * (W + 2) + ((r & 1) ? W + 1 : 0);
            act[p * (int64_t)(H + 2) * (W + 2) + px] = make_uint4(0, 0, 0, 0);
        }
        return;
    }
    convert_weights<false>(n.w[l], wimg + n.off[l], n.CI[l], n.CO[l], n.NT[l]);
}

// Input rows i0 - 1 .. i0 + kHaloRows of channel block cb, pixels j0 - 1 ..
// j0 + 128, as BF16 (zeros outside the image and past CI): 16-byte row
// ((row * 4 + channel group) * kHaloQ + pixel). Consecutive threads take
// consecutive pixels, so each of the 8 loads of a row is coalesced; all of a
// thread's 40 loads are in flight together. WIDE = false: a block's 32 planes
// span less than 4 GB, so a load's address is a base shared by the CTA plus the
// thread's 32-bit offset. At 4.8 TB/s from L2 (the halo rows are read twice over)
// the staging bounds the kernel.
template <bool WIDE>
__device__ __forceinline__ void stage_halo(unsigned char *hb, const float *__restrict__ xn, int cb, int CI, int H,
                                           int W, int i0, int j0)
{
    constexpr int items = (kHaloRows + 2) * (kHaloCB / 8) * kHaloQ, per = items / (32 * kProdWarps);
    static_assert(per * 32 * kProdWarps == items, "every thread takes the same number of rows");
    const int64_t HW = (int64_t)H * W;
    const int c0 = cb * kHaloCB;
    const char *base = reinterpret_cast<const char *>(xn + (int64_t)c0 * HW + (int64_t)(i0 - 1) * W + (j0 - 1));
    float v[per][8];
#pragma unroll
    for (int z = 0; z < per; ++z) {
        const int it = threadIdx.x + z * 32 * kProdWarps;
        const int q = it % kHaloQ, rest = it / kHaloQ;
        const int g = rest % (kHaloCB / 8), rr = rest / (kHaloCB / 8);
        const bool in = (unsigned)(i0 - 1 + rr) < (unsigned)H && (unsigned)(j0 - 1 + q) < (unsigned)W;
        const int nc = in ? CI - c0 - 8 * g : 0;
        const int64_t o64 = 4 * (8 * g * HW + (int64_t)rr * W + q);
        const unsigned o32 = 4u * (8u * (unsigned)g * (unsigned)HW + (unsigned)(rr * W + q));
        if (nc >= 8) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                v[z][e] = __ldg(reinterpret_cast<const float *>(base + 4 * e * HW + (WIDE ? o64 : (int64_t)o32)));
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                v[z][e] = e < nc ? __ldg(reinterpret_cast<const float *>(base + 4 * e * HW + (WIDE ? o64 : (int64_t)o32))) : 0.f;
        }
    }
#pragma unroll
    for (int z = 0; z < per; ++z) {
        uint32_t pk[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) pk[e] = bf16_pair(v[z][2 * e], v[z][2 * e + 1]);
        *reinterpret_cast<uint4 *>(hb + (size_t)(threadIdx.x + z * 32 * kProdWarps) * 16) =
            make_uint4(pk[0], pk[1], pk[2], pk[3]);
    }
}

// nh staging buffers and nw weight slots (nw = all of the layer's blocks when
// they are resident; then there is one block of output channels). relu: write
// max(y, 0).
//
// Between the layers of one call (dg_nn_forward_tc) the activations wait as the
// BF16 values the products take, already rounded as the staging rounds them (the
// same results bit for bit), in the staging's own layout: IN16 / OUT16 tensors are
// [image][channels / 8][H + 2][W + 2][8] with a border of zeros, channels a
// multiple of 32. A staged row is then one bulk copy of consecutive bytes, and an
// output pixel's 32 channels are four 16-byte stores: no conversion, half the bytes
// and no registers on the way in (network at 512 x 512: 238 -> 145 us).
template <bool WIDE, bool IN16, bool OUT16>
__global__ void __launch_bounds__(kConvThreads, 1)
    k_conv3x3_tc(const void *__restrict__ xv, const uint16_t *__restrict__ wimg, const float *__restrict__ b,
                 void *__restrict__ yv, int CI, int CO, int H, int W, int NT, int nh, int nw, int64_t tiles, int relu,
                 unsigned *err)
{
    extern __shared__ __align__(1024) unsigned char nsm[];
    __shared__ __align__(8) uint64_t wfull[kWSlots], wempty[kWSlots], hfull[kHaloMax], hempty[kHaloMax], afull[2],
        aempty[2], fin;
    __shared__ uint32_t tslot;
    const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
    const int ob = (CO + NT - 1) / NT;
    const int ncb = (CI + kHaloCB - 1) / kHaloCB, nblk = ncb * 9;
    const int tx = (W + kRowsTc - 1) / kRowsTc, ty = (H + kHaloRows - 1) / kHaloRows;
    const bool resident = nw == nblk && ob == 1;
    const int AS = acc_stride(NT);
    const uint32_t wbytes = (uint32_t)NT * kHaloCB * 2;
    const uint32_t ncols = (uint32_t)tmem_cols(2 * kHaloRows * AS);
    unsigned char *wring = nsm + (size_t)nh * kHaloBytes;
    struct Tile {
        int n, obi, i0, j0;
    };
    const float *x = reinterpret_cast<const float *>(xv);
    float *y = reinterpret_cast<float *>(yv);
    const int64_t plane = (int64_t)(H + 2) * (W + 2) * 16;  // bytes of 8 channels of a BF16 tensor
    auto tile_of = [&](int64_t v) {
        Tile o;
        o.j0 = (int)(v % tx) * kRowsTc;
        v /= tx;
        o.i0 = (int)(v % ty) * kHaloRows;
        v /= ty;
        o.obi = (int)(v % ob);
        o.n = (int)(v / ob);
        return o;
    };
    if (t == 0) {
        for (int k = 0; k < nw; ++k) {
            nn_mbar_init(smem_addr(&wfull[k]), 1);
            nn_mbar_init(smem_addr(&wempty[k]), 1);
        }
        for (int k = 0; k < nh; ++k) {
            nn_mbar_init(smem_addr(&hfull[k]), IN16 ? 1 : kProdWarps);
            nn_mbar_init(smem_addr(&hempty[k]), 1);
        }
        for (int k = 0; k < 2; ++k) {
            nn_mbar_init(smem_addr(&afull[k]), 1);
            nn_mbar_init(smem_addr(&aempty[k]), kOutWarps);
        }
        nn_mbar_init(smem_addr(&fin), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) nn_tmem_alloc(smem_addr(&tslot), ncols);
    nn_before_sync();
    __syncthreads();
    nn_after_sync();
    const uint32_t tmem = tslot;
    // Everything above runs while the kernel before still drains (launch_waiting);
    // its outputs, and what this one overwrites, are safe from here on. Dependents are let in only after
    // that wait, so a kernel's predecessors but one have always finished.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool ok = true;
    int64_t copied = 0;  // weight blocks (or BF16 input stages) whose copies this thread has issued
    if (IN16 && warp < kProdWarps) {
        if (warp == 0) {
            int s = 0;
            uint32_t ph = 1;
            for (int64_t v = blockIdx.x; v < tiles && ok; v += gridDim.x) {
                const Tile o = tile_of(v);
                const int rows = min(kHaloRows + 2, H + 2 - o.i0);  // those of the bordered image
                const uint32_t len = (uint32_t)min(kHaloQ, W + 2 - o.j0) * 16;
                const int rr = lane / (kHaloCB / 8), g = lane % (kHaloCB / 8);
                const char *src = reinterpret_cast<const char *>(xv) + (int64_t)o.n * (CI / 8) * plane + (int64_t)g * plane +
                                  ((int64_t)(o.i0 + rr) * (W + 2) + o.j0) * 16;
                for (int cb = 0; cb < ncb; ++cb, src += (kHaloCB / 8) * plane) {
                    ok = __all_sync(0xffffffffu, nn_wait(smem_addr(&hempty[s]), ph));
                    if (!ok) break;
                    if (lane == 0) {
                        nn_expect_tx(smem_addr(&hfull[s]), (uint32_t)(rows * (kHaloCB / 8)) * len);
                        ++copied;
                    }
                    __syncwarp();
                    if (rr < rows)
                        nn_bulk_g2s(smem_addr(nsm + (size_t)s * kHaloBytes + (size_t)lane * kHaloQ * 16), src, len,
                                    smem_addr(&hfull[s]));
                    if (++s == nh) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
        }
    } else if (warp < kProdWarps) {
        int s = 0;
        uint32_t ph = 1;  // parity of the buffer's last release; a fresh barrier passes parity 1
        for (int64_t v = blockIdx.x; v < tiles && ok; v += gridDim.x) {
            const Tile o = tile_of(v);
            const float *xn = x + (size_t)o.n * CI * H * W;
            for (int cb = 0; cb < ncb; ++cb) {
                ok = nn_wait(smem_addr(&hempty[s]), ph);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                stage_halo<WIDE>(nsm + (size_t)s * kHaloBytes, xn, cb, CI, H, W, o.i0, o.j0);
                nn_fence_async();
                __syncwarp();
                if (lane == 0) nn_arrive(smem_addr(&hfull[s]));
                if (++s == nh) {
                    s = 0;
                    ph ^= 1;
                }
            }
        }
    } else if (warp < kProdWarps + kOutWarps) {
        // tensor-memory lanes (pixels) 32 q .. + 31, output row r of the tile
        const int q = warp & 3, r = (warp - kProdWarps) >> 2;
        int set = 0;
        uint32_t ph = 0;
        for (int64_t v = blockIdx.x; v < tiles && ok; v += gridDim.x) {
            const Tile o = tile_of(v);
            ok = __all_sync(0xffffffffu, nn_wait(smem_addr(&afull[set]), ph));
            if (!ok) break;
            nn_after_sync();
            const int jp = o.j0 + 32 * q + lane, o0 = o.obi * NT;
            float *yn = y + (size_t)o.n * CO * H * W;
            const int64_t HW = (int64_t)H * W;
            const int i = o.i0 + r;
            const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)((set * kHaloRows + r) * AS);
            const unsigned o32 = 4u * (unsigned)(i * W + jp);
            for (int c0 = 0; c0 < NT; c0 += 32) {
                uint32_t rv[32];
                nn_ld32(tl + (uint32_t)c0, rv);
                const int nc = min(min(NT - c0, CO - o0 - c0), 32);
                const float bl = b && lane < nc ? __ldg(b + o0 + c0 + lane) : 0.f;
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    const float val = __uint_as_float(rv[e]) + __shfl_sync(0xffffffffu, bl, e);
                    rv[e] = __float_as_uint(relu ? fmaxf(val, 0.f) : val);
                }
                if (OUT16) {
                    if (i < H && jp < W) {
                        char *dst = reinterpret_cast<char *>(yv) + ((int64_t)o.n * (CO / 8) + (o0 + c0) / 8) * plane +
                                    ((int64_t)(i + 1) * (W + 2) + jp + 1) * 16;
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            uint32_t pk[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                pk[e] = bf16_pair(__uint_as_float(rv[8 * g + 2 * e]), __uint_as_float(rv[8 * g + 2 * e + 1]));
                            if (8 * g < nc) *reinterpret_cast<uint4 *>(dst + g * plane) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        }
                    }
                } else if (i < H && jp < W) {
                    char *dst = reinterpret_cast<char *>(yn + (int64_t)(o0 + c0) * HW);
                    const int64_t off = WIDE ? 4 * ((int64_t)i * W + jp) : (int64_t)o32;
                    if (nc == 32) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) *reinterpret_cast<float *>(dst + 4 * e * HW + off) = __uint_as_float(rv[e]);
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (e < nc) *reinterpret_cast<float *>(dst + 4 * e * HW + off) = __uint_as_float(rv[e]);
                    }
                }
            }
            nn_before_sync();
            __syncwarp();
            if (lane == 0) nn_arrive(smem_addr(&aempty[set]));
            if (set) ph ^= 1;
            set ^= 1;
        }
    } else if (warp == kProdWarps + kOutWarps) {
        if (lane == 0) {
            int slot = 0;
            uint32_t ph = 1;
            for (int64_t v = blockIdx.x; v < tiles && ok; v += gridDim.x) {
                const unsigned char *wsrc = reinterpret_cast<const unsigned char *>(wimg) +
                                            (size_t)tile_of(v).obi * nblk * wbytes;
                for (int g = 0; g < nblk && ok; ++g) {
                    ok = nn_wait(smem_addr(&wempty[slot]), ph);
                    if (!ok) break;
                    nn_expect_tx(smem_addr(&wfull[slot]), wbytes);
                    nn_bulk_g2s(smem_addr(wring + (size_t)slot * wbytes), wsrc + (size_t)g * wbytes, wbytes,
                                smem_addr(&wfull[slot]));
                    ++copied;
                    if (++slot == nw) {
                        slot = 0;
                        ph ^= 1;
                    }
                }
                if (resident) break;
            }
        }
    } else {
        const uint32_t lead = nn_elect(), id = nn_idesc(NT);
        int s = 0, slot = 0, set = 0;
        uint32_t hph = 0, wph = 0, aph = 1;
        bool first = true;
        for (int64_t v = blockIdx.x; v < tiles && ok; v += gridDim.x) {
            ok = __all_sync(0xffffffffu, nn_wait(smem_addr(&aempty[set]), aph));
            const uint32_t acc0 = tmem + (uint32_t)(set * kHaloRows * AS);
            for (int cb = 0; cb < ncb && ok; ++cb) {
                ok = __all_sync(0xffffffffu, nn_wait(smem_addr(&hfull[s]), hph));
                if (!ok) break;
                const uint64_t ad = halo_desc(smem_addr(nsm) + (uint32_t)(s * kHaloBytes));
#pragma unroll
                for (int tap = 0; tap < 9; ++tap) {
                    if (first || !resident) {
                        ok = ok && nn_wait(smem_addr(&wfull[slot]), wph);
                        ok = __all_sync(0xffffffffu, ok);
                    }
                    nn_after_sync();
                    if (ok) {
                        const int u = tap / 3, vv = tap - 3 * (tap / 3);
                        const uint64_t wd = nn_sdesc(smem_addr(wring) + (uint32_t)slot * wbytes);
#pragma unroll
                        for (int r = 0; r < kHaloRows; ++r)
#pragma unroll
                            for (int h = 0; h < kHaloCB / 16; ++h)
                                nn_mma_if(lead, acc0 + (uint32_t)(r * AS),
                                          ad + (uint64_t)(((r + u) * (kHaloCB / 8) + 2 * h) * kHaloQ + vv),
                                          wd + (uint64_t)(16 * h), id, (cb > 0 || tap > 0 || h > 0) ? 1u : 0u);
                        if (!resident && lead) nn_commit(smem_addr(&wempty[slot]));
                    }
                    if (++slot == nw) {
                        slot = 0;
                        wph ^= 1;
                    }
                }
                if (lead) nn_commit(smem_addr(&hempty[s]));
                if (++s == nh) {
                    s = 0;
                    hph ^= 1;
                }
            }
            if (lead) nn_commit(smem_addr(&afull[set]));
            first = false;
            if (set) aph ^= 1;
            set ^= 1;
        }
        // completes once every MMA issued is done
        if (lead) nn_commit(smem_addr(&fin));
    }
    __syncwarp();
    // before tensor memory and shared memory are released the MMAs and copies
    // issued have landed, also where a wait gave up
    if (IN16 && t == 0)
        for (int64_t g = copied > nh ? copied - nh : 0; g < copied; ++g)
            ok = nn_wait(smem_addr(&hfull[g % nh]), (uint32_t)(g / nh) & 1u) && ok;
    if (t == 32 * (kProdWarps + kOutWarps))
        for (int64_t g = copied > nw ? copied - nw : 0; g < copied; ++g)
            ok = nn_wait(smem_addr(&wfull[g % nw]), (uint32_t)(g / nw) & 1u) && ok;
    ok = __syncthreads_and(ok) != 0;
    if (t == 0) {
        ok = nn_wait(smem_addr(&fin), 0u) && ok;
        if (!ok) atomicOr(err, 1u);
    }
    nn_before_sync();
    __syncthreads();
    nn_after_sync();
    if (warp == 0) nn_tmem_free(tmem, ncols);
}

// ---------------------------------------------------------------------------
// Weight and bias gradient: K = pixels, rows = output channels (CO <= 128),
// columns = 32 input channels, one accumulator per tap (9 x 32 of the 512
// tensor-memory columns).
//
// Both operands are staged as the forward's halo is: 16-byte rows of 8
// channels of one pixel, consecutive pixels 16 B apart. Read with the channel
// dimension as M / N and the pixels as K that is the canonical MN-major
// layout (core matrix: 8 pixels x 8 channels, 128 B along the pixels, the
// channel groups a row of pixels apart), so the x operand of tap (u, v) is the
// same staged row seen v pixels further, and u is one of three staged rows:
// nothing is gathered per tap. (With pixels contiguous in each row, the K-major
// layout, a shift by one pixel is no aligned start; the gathers it took, 9
// loads per element, were 2.05 ms of the 2.33 ms of a 64 -> 128 channel
// backward at 16 x 128 x 128.)
// A CTA walks output rows of `tw` pixels (i fastest) of one block of 32 input
// channels: dy in two buffers, x rows in a ring of four. 16 warps load the next
// row's dy and its one new x row into registers a whole step ahead and store
// them rounded, while one more warp issues the current row's 9 x tw / 16 MMAs.
// That warp runs its loop with all lanes (nn_elect): issued from a branch on one
// thread an MMA took 130 cycles, most of them moving descriptors into uniform
// registers, and the kernel 155 us at that size; now 82 us, bound by the 80 KB a
// row that each CTA loads and converts (8 staging warps: 125 us). Channel groups
// are padded by one pixel against bank conflicts. Partial sums:
// part[split][tap][c][o], then the bias [split][o].
// ---------------------------------------------------------------------------
constexpr int kDwThreads = 512;                // staging threads; one more warp issues the MMAs
constexpr int kDwCB = 32;                      // input channels per CTA
constexpr int kDwRing = 4;                     // staged x rows

// bytes of one dy buffer, of one x row
__host__ __device__ constexpr int dw_a_bytes(int tw) { return (kRowsTc / 8) * (tw + 1) * 16; }
__host__ __device__ constexpr int dw_x_bytes(int tw) { return (kDwCB / 8) * (tw + 2) * 16; }
__host__ __device__ constexpr int dw_smem(int tw) { return 2 * dw_a_bytes(tw) + kDwRing * dw_x_bytes(tw); }

// MN-major, no swizzle: pixel groups (K) 128 B apart (leading byte offset),
// channel groups (M / N) `group` B apart (stride byte offset)
__device__ __forceinline__ uint64_t mn_desc(uint32_t saddr, uint32_t group)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(group >> 4) << 32) |
           (1ull << 46);
}

__device__ __forceinline__ uint4 pack8(const float (&v)[8])
{
    uint32_t pk[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) pk[e] = bf16_pair(v[2 * e], v[2 * e + 1]);
    return make_uint4(pk[0], pk[1], pk[2], pk[3]);
}

__global__ void __launch_bounds__(kDwThreads + 32, 1)
    k_conv3x3_dw_tc(const float *__restrict__ x, const float *__restrict__ dy, float *__restrict__ part, int CI, int CO,
                    int H, int W, int tw, int nb, int64_t rows, int64_t per_split, int S, unsigned *err)
{
    extern __shared__ __align__(1024) unsigned char nsm[];
    __shared__ __align__(8) uint64_t done[2];
    __shared__ uint32_t tslot;
    const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
    const bool mma_warp = warp == kDwThreads / 32;  // ng <= 16 groups: no bias there
    const int c0 = blockIdx.x * kDwCB, split = blockIdx.y;
    const int64_t r_lo = (int64_t)split * per_split, r_hi = min(rows, r_lo + per_split);
    const int nrow = r_hi > r_lo ? (int)(r_hi - r_lo) : 0;
    const int abytes = dw_a_bytes(tw), xbytes = dw_x_bytes(tw), xq = tw + 2;
    unsigned char *sa = nsm, *sx = nsm + 2 * abytes;
    const int64_t HW = (int64_t)H * W;
    if (t == 0) {
        nn_mbar_init(smem_addr(&done[0]), 1);
        nn_mbar_init(smem_addr(&done[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) nn_tmem_alloc(smem_addr(&tslot), 512u);
    // rows of output channels past CO are zero in both dy buffers
    for (int i = t; i < 2 * abytes / 16; i += kDwThreads + 32)
        *reinterpret_cast<uint4 *>(sa + 16 * (size_t)i) = make_uint4(0, 0, 0, 0);
    nn_before_sync();
    __syncthreads();
    nn_after_sync();
    const uint32_t tmem = tslot;
    // FP32 D, BF16 A and B, both MN-major, N = 32, M = 128
    const uint32_t id = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(kDwCB >> 3) << 17) |
                        ((uint32_t)(kRowsTc >> 4) << 24);
    const int ng = (CO + 7) / 8;  // groups of 8 output channels
    struct Row {  // image, first column, row of a step
        int n, j0, i;
    };
    auto next = [&](Row &o) {
        if (++o.i == H) {
            o.i = 0;
            o.j0 += tw;
            if (o.j0 >= nb * tw) {
                o.j0 = 0;
                ++o.n;
            }
        }
    };
    Row cur;  // the only divisions
    cur.i = (int)(r_lo % H);
    cur.j0 = (int)((r_lo / H) % nb) * tw;
    cur.n = (int)(r_lo / H / nb);
    // x row `row` of the strip (zero outside the image): into registers, and
    // into its ring slot
    constexpr int kXi = ((kDwCB / 8) * (kRowsTc + 2) + kDwThreads - 1) / kDwThreads;
    float xv[kXi][8];
    int xo[kXi], xcol[kXi], xch[kXi];  // this thread's pixels: offset of 8 channels, column and first channel
#pragma unroll
    for (int k = 0; k < kXi; ++k) {
        const int it = t + k * kDwThreads;
        xcol[k] = it % xq - 1;
        xch[k] = it / xq < kDwCB / 8 ? c0 + 8 * (it / xq) : CI;
        xo[k] = 16 * it;
    }
    auto load_x = [&](const Row &o, int row) {
        const bool in = row >= 0 && row < H;
#pragma unroll
        for (int k = 0; k < kXi; ++k) {
            const int col = o.j0 + xcol[k], nc = in && col >= 0 && col < W ? CI - xch[k] : 0;
            const float *src = x + ((int64_t)o.n * CI + xch[k]) * HW + (int64_t)row * W + col;
            if (nc >= 8) {
#pragma unroll
                for (int e = 0; e < 8; ++e) xv[k][e] = __ldg(src + e * HW);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) xv[k][e] = e < nc ? __ldg(src + e * HW) : 0.f;
            }
        }
    };
    auto store_x = [&](int row) {
        unsigned char *dst = sx + (size_t)(row & (kDwRing - 1)) * xbytes;
#pragma unroll
        for (int k = 0; k < kXi; ++k)
            if (xo[k] < xbytes) *reinterpret_cast<uint4 *>(dst + xo[k]) = pack8(xv[k]);
    };
    // dy: item k of a warp is a group of 8 channels x 32 pixels, lanes along the pixels
    constexpr int kDi = (kRowsTc / 8) * (kRowsTc / 32) / (kDwThreads / 32);
    float v[kDi][8];
    auto load_dy = [&](const Row &o) {
        const int left = min(tw, W - o.j0);
        const float *base = dy + (int64_t)o.n * CO * HW + (int64_t)o.i * W + o.j0;
#pragma unroll
        for (int k = 0; k < kDi; ++k) {
            const int it = warp + k * (kDwThreads / 32), q = 32 * (it & 3) + lane, g = it >> 2;
            const int nc = q < left ? min(8, CO - 8 * g) : 0;
            const float *src = base + (int64_t)8 * g * HW + q;
            if (nc >= 8) {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[k][e] = __ldg(src + e * HW);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[k][e] = e < nc ? __ldg(src + e * HW) : 0.f;
            }
        }
    };
    auto store_dy = [&](int buf) {
#pragma unroll
        for (int k = 0; k < kDi; ++k) {
            const int it = warp + k * (kDwThreads / 32), q = 32 * (it & 3) + lane, g = it >> 2;
            if (g < ng && q < tw)
                *reinterpret_cast<uint4 *>(sa + (size_t)buf * abytes + ((size_t)g * (tw + 1) + q) * 16) = pack8(v[k]);
        }
    };
    // the registers hold the next row's dy and its one new x row, loaded a whole
    // step before they are stored
    Row pre = cur;  // the row in the registers
    if (nrow > 1) next(pre);
    if (nrow > 0 && !mma_warp) {
        for (int u = -1; u <= 0; ++u) {
            load_x(cur, cur.i + u);
            store_x(cur.i + u);
        }
        load_dy(cur);
        load_x(cur, cur.i + 1);
        store_x(cur.i + 1);
        store_dy(0);
        nn_fence_async();
        if (nrow > 1) {
            load_dy(pre);
            load_x(pre, pre.i + 1);
        }
    }
    float db8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // bias: warp w sums channels 8 w .. 8 w + 7
    bool ok = __syncthreads_and(1) != 0;
    int issued = 0;  // rows whose MMAs have been issued
    for (int k = 0; k < nrow && ok; ++k) {
        issued = k + 1;
        if (mma_warp) {
            nn_after_sync();
            const uint32_t lead = nn_elect();
            const uint64_t da = mn_desc(smem_addr(sa) + (uint32_t)((k & 1) * abytes), (uint32_t)(tw + 1) * 16);
            const uint32_t xb = smem_addr(sx);
            for (int ks = 0; ks < tw / 16; ++ks) {  // 256 bytes further per 16 pixels
                const uint32_t acc = (k > 0 || ks > 0) ? 1u : 0u;
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                    const uint64_t db = mn_desc(xb + (uint32_t)(((cur.i + u - 1) & (kDwRing - 1)) * xbytes), (uint32_t)xq * 16);
#pragma unroll
                    for (int vv = 0; vv < 3; ++vv)
                        nn_mma_if(lead, tmem + (uint32_t)((3 * u + vv) * kDwCB), da + (uint64_t)(16 * ks),
                                  db + (uint64_t)(16 * ks + vv), id, acc);
                }
            }
            if (lead) nn_commit(smem_addr(&done[k & 1]));
            __syncwarp();
        } else if (k + 1 < nrow) {
            // the buffers written next were read by the MMAs of row k - 1; a new
            // strip replaces rows that row k's MMAs read
            const bool strip = pre.i == 0;
            if (strip) ok = nn_wait(smem_addr(&done[k & 1]), (uint32_t)(k >> 1) & 1u);
            else if (k > 0) ok = nn_wait(smem_addr(&done[(k - 1) & 1]), (uint32_t)((k - 1) >> 1) & 1u);
            if (ok) {
                store_x(pre.i + 1);
                store_dy((k + 1) & 1);
                if (strip)
                    for (int u = -1; u <= 0; ++u) {
                        load_x(pre, u);
                        store_x(u);
                    }
                nn_fence_async();
            }
        }
        cur = pre;
        if (k + 2 < nrow) {
            next(pre);
            if (!mma_warp) {
                load_dy(pre);
                load_x(pre, pre.i + 1);
            }
        }
        if (blockIdx.x == 0 && warp < ng)  // the staged (rounded) row, on the CUDA cores
            for (int q = lane; q < tw; q += 32) {
                const uint4 p = *reinterpret_cast<const uint4 *>(sa + (size_t)(k & 1) * abytes +
                                                                 ((size_t)warp * (tw + 1) + q) * 16);
                const uint32_t w4[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    db8[2 * e] += __uint_as_float(w4[e] << 16);
                    db8[2 * e + 1] += __uint_as_float(w4[e] & 0xffff0000u);
                }
            }
        nn_before_sync();
        ok = __syncthreads_and(ok) != 0;
    }
    // the last commits cover every MMA issued (also after a wait gave up)
    for (int k = max(0, issued - 2); k < issued; ++k) {
        const bool fin = nn_wait(smem_addr(&done[k & 1]), (uint32_t)(k >> 1) & 1u);
        ok = ok && fin;
    }
    ok = __syncthreads_and(ok) != 0;
    nn_after_sync();
    if (!ok) {
        if (t == 0) atomicOr(err, 1u);
    } else {
        if (warp < 4) {  // warp w holds output channels 32 w .. 32 w + 31
            const int o = 32 * warp + lane;
            const uint32_t tl = tmem + ((uint32_t)(32 * warp) << 16);
            for (int tap = 0; tap < 9; ++tap) {
                uint32_t r[32];
                nn_ld32(tl + (uint32_t)(tap * kDwCB), r);
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    if (o < CO && c0 + e < CI)
                        part[(((size_t)split * 9 + tap) * CI + c0 + e) * CO + o] = nrow > 0 ? __uint_as_float(r[e]) : 0.f;
            }
        }
        if (blockIdx.x == 0 && warp < ng) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float b = db8[e];
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) b += __shfl_xor_sync(0xffffffffu, b, d);
                if (lane == 0 && 8 * warp + e < CO) part[(size_t)S * 9 * CI * CO + (size_t)split * CO + 8 * warp + e] = b;
            }
        }
    }
    nn_before_sync();
    __syncthreads();
    nn_after_sync();
    if (warp == 0) nn_tmem_free(tmem, 512u);
}

// dw[o][c][u][v] and db[o] = the splits' partial sums, added in split order.
__global__ void k_conv3x3_dw_tc_sum(const float *__restrict__ part, float *__restrict__ dw, float *__restrict__ db,
                                    int CI, int CO, int S)
{
    const int64_t n = (int64_t)9 * CI * CO;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n + CO; e += (int64_t)gridDim.x * blockDim.x) {
        const float *p = e < n ? part + e : part + (size_t)S * n + (e - n);
        const int64_t stride = e < n ? n : CO;
        float acc = 0.f;
#pragma unroll 8
        for (int s = 0; s < S; ++s) acc += __ldg(p + (size_t)s * stride);
        if (e < n) {
            const int o = (int)(e % CO), c = (int)((e / CO) % CI), tap = (int)(e / ((int64_t)CO * CI));
            dw[((size_t)o * CI + c) * 9 + tap] = acc;
        } else {
            db[e - n] = acc;
        }
    }
}

__device__ unsigned g_nn_tc_err;  // a tensor-core layer's wait gave up (dg_nn_tc_check)

namespace {

int nt_of(int co) { return std::min(128, (co + 15) / 16 * 16); }
// Pixels of an output row per step (a multiple of 16, at most 128, the row in
// equal parts), parts per row, and splits: one CTA per SM over the blocks of
// input channels, a row each at least.
struct DwShape {
    int tw, nb;
    int64_t rows, S;
};
DwShape dw_shape(int B, int Ci, int H, int W)
{
    DwShape d;
    d.nb = (W + kRowsTc - 1) / kRowsTc;
    d.tw = ((W + d.nb - 1) / d.nb + 15) / 16 * 16;
    d.rows = (int64_t)B * H * d.nb;
    const int64_t blocks = (Ci + kDwCB - 1) / kDwCB;
    d.S = std::max<int64_t>(1, std::min<int64_t>(d.rows, std::max<int64_t>(1, 152 / blocks)));
    return d;
}

bool tc_shape_ok(int B, int Ci, int Co, int H, int W)
{
    return B > 0 && Ci > 0 && Co > 0 && H > 0 && W > 0 && Ci <= 4096 && Co <= 4096 && H <= 65535 &&
           (int64_t)B * ((Co + 127) / 128) <= 65535 && (int64_t)B * std::max(Ci, Co) * H * W <= ((int64_t)1 << 40);
}

unsigned *err_word()
{
    void *p = nullptr;
    return cudaGetSymbolAddress(&p, g_nn_tc_err) == cudaSuccess ? (unsigned *)p : nullptr;
}

// Launch of a kernel that itself waits for the one before it in the stream
// (griddepcontrol.wait), so that its setup and its launch overlap that one's end: the
// five layers of the proposal network 145 -> 132 us.
template <typename... P, typename... A>
cudaError_t launch_waiting(void (*kernel)(P...), dim3 grid, int threads, int smem, cudaStream_t s, A... args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// The convolution on converted weights.
cudaError_t launch_conv_blocks(const void *x, const uint16_t *wimg, const float *b, void *y, int B, int CI, int CO, int H,
                               int W, cudaStream_t s, int relu, bool in16 = false, bool out16 = false)
{
    unsigned *err = err_word();
    if (!err) return cudaErrorInvalidSymbol;
    const int NT = nt_of(CO);
    cudaError_t e;
    // the whole layer's weights beside at least two staging buffers, or else a
    // ring of 16 slots at most
    const int ob = (CO + NT - 1) / NT, nblk = (CI + kHaloCB - 1) / kHaloCB * 9, wbytes = NT * kHaloCB * 2;
    const bool resident = ob == 1 && nblk <= kWSlots && nblk * wbytes + 2 * kHaloBytes <= kConvSmem;
    const int nw = resident ? nblk : std::min(nblk, std::min(16, (kConvSmem - 2 * kHaloBytes) / wbytes));
    const int nh = std::min(kHaloMax, (kConvSmem - nw * wbytes) / kHaloBytes);
    const int smem = nh * kHaloBytes + nw * wbytes;
    // 32 planes and a row of pixels each, in bytes, against the 32-bit offsets
    const bool wide = 4.0 * (kHaloCB * (double)H * W + 8.0 * W + 4096.0) > 4294967295.0;
    auto kernel = in16 ? (out16 ? (wide ? k_conv3x3_tc<true, true, true> : k_conv3x3_tc<false, true, true>)
                                : (wide ? k_conv3x3_tc<true, true, false> : k_conv3x3_tc<false, true, false>))
                       : (out16 ? (wide ? k_conv3x3_tc<true, false, true> : k_conv3x3_tc<false, false, true>)
                                : (wide ? k_conv3x3_tc<true, false, false> : k_conv3x3_tc<false, false, false>));
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess)
        return e;
    const int64_t tiles = (int64_t)((W + kRowsTc - 1) / kRowsTc) * ((H + kHaloRows - 1) / kHaloRows) * B * ob;
    return launch_waiting(kernel, dim3((unsigned)std::min<int64_t>(tiles, 152)), kConvThreads, smem, s, x, wimg, b, y, CI, CO, H,
                          W, NT, nh, nw, tiles, relu, err);
}

cudaError_t launch_conv_tc(bool tr, const float *x, const float *w, const float *b, float *y, int B, int CI, int CO,
                           int H, int W, uint16_t *wimg, cudaStream_t s, int relu = 0)
{
    const int NT = nt_of(CO);
    const int64_t items = wimg_elems(CI, CO, NT) / 8;
    const unsigned gw = (unsigned)std::min<int64_t>((items + 255) / 256, 152 * 8);
    if (tr) k_conv_tc_wimg<true><<<gw, 256, 0, s>>>(w, wimg, CI, CO, NT);
    else k_conv_tc_wimg<false><<<gw, 256, 0, s>>>(w, wimg, CI, CO, NT);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_conv_blocks(x, wimg, b, y, B, CI, CO, H, W, s, relu);
}

// Whether a network's hidden layers wait as BF16 tensors (k_conv3x3_tc).
bool net16(const int32_t *ch, int L)
{
    for (int l = 1; l < L; ++l)
        if (ch[l] % kHaloCB) return false;
    return L > 1;
}

// Scratch of a whole network (floats): every layer's blocks, then two buffers of
// the widest hidden layer (act floats each); off: the layers' blocks (elements). -1:
// a shape out of range.
int64_t net_scratch(const int32_t *ch, int L, int B, int H, int W, int64_t *off, int64_t *act)
{
    if (!ch || L < 1 || L > kNetLayers) return -1;
    int64_t e = 0;
    int wide = 0;
    for (int l = 0; l < L; ++l) {
        if (!tc_shape_ok(B, ch[l], ch[l + 1], H, W)) return -1;
        if (off) off[l] = e;
        e += (wimg_elems(ch[l], ch[l + 1], nt_of(ch[l + 1])) + 7) / 8 * 8;
        if (l > 0) wide = std::max(wide, ch[l]);
    }
    const int64_t a = net16(ch, L) ? (int64_t)B * (wide / 8) * (H + 2) * (W + 2) * 4 : ((int64_t)B * wide * H * W + 3) / 4 * 4;
    if (act) *act = a;
    return e / 2 + (L > 2 ? 2 : L > 1 ? 1 : 0) * a;
}

// floats of scratch: the forward's weight blocks, or the backward's (data
// gradient weight blocks, then the weight gradient's partial sums)
int64_t fwd_scratch(int Ci, int Co) { return (wimg_elems(Ci, Co, nt_of(Co)) + 7) / 8 * 4; }
int64_t bwd_wimg_floats(int Ci, int Co) { return (wimg_elems(Co, Ci, nt_of(Ci)) + 7) / 8 * 4; }

}  // namespace

int64_t nn_conv_tc_scratch(int B, int Ci, int Co, int H, int W)
{
    return std::max(fwd_scratch(Ci, Co), bwd_wimg_floats(Ci, Co) + dw_shape(B, Ci, H, W).S * (int64_t)Co * (Ci * 9 + 1));
}

}  // namespace dg

extern "C" {

static dg_status conv_forward_tc(const char *name, const float *x, const float *w, const float *b, float *y, int32_t B,
                                 int32_t Ci, int32_t Co, int32_t H, int32_t W, float *scratch, void *stream, int relu)
{
    if (!x || !w || !b || !y || !scratch) return dg::nn_fail(DG_EINVAL, "%s: null pointer", name);
    if (!dg::tc_shape_ok(B, Ci, Co, H, W))
        return dg::nn_fail(DG_EINVAL, "%s: bad shape B=%d Ci=%d Co=%d H=%d W=%d", name, B, Ci, Co, H, W);
    if ((reinterpret_cast<uintptr_t>(scratch) & 15) != 0)
        return dg::nn_fail(DG_EINVAL, "%s: scratch must be 16-byte aligned", name);
    return dg::nn_done(dg::launch_conv_tc(false, x, w, b, y, B, Ci, Co, H, W, reinterpret_cast<uint16_t *>(scratch),
                                          (cudaStream_t)stream, relu),
                       name);
}

dg_status dg_nn_conv3x3_forward_tc(const float *x, const float *w, const float *b, float *y, int32_t B, int32_t Ci,
                                   int32_t Co, int32_t H, int32_t W, float *scratch, void *stream)
{
    return conv_forward_tc("dg_nn_conv3x3_forward_tc", x, w, b, y, B, Ci, Co, H, W, scratch, stream, 0);
}

dg_status dg_nn_conv3x3_relu_forward_tc(const float *x, const float *w, const float *b, float *y, int32_t B, int32_t Ci,
                                        int32_t Co, int32_t H, int32_t W, float *scratch, void *stream)
{
    return conv_forward_tc("dg_nn_conv3x3_relu_forward_tc", x, w, b, y, B, Ci, Co, H, W, scratch, stream, 1);
}

int64_t dg_nn_forward_tc_scratch(const int32_t *channels, int32_t layers, int32_t B, int32_t H, int32_t W)
{
    return dg::net_scratch(channels, layers, B, H, W, nullptr, nullptr);
}

dg_status dg_nn_forward_tc(const float *x, const float *const *w, const float *const *b, const int32_t *channels,
                           int32_t layers, float *y, int32_t B, int32_t H, int32_t W, float *scratch, void *stream)
{
    if (!x || !w || !b || !channels || !y || !scratch) return dg::nn_fail(DG_EINVAL, "dg_nn_forward_tc: null pointer");
    int64_t act = 0;
    dg::NetWeights n{};
    if (dg::net_scratch(channels, layers, B, H, W, n.off, &act) < 0)
        return dg::nn_fail(DG_EINVAL, "dg_nn_forward_tc: bad shape (%d layers, B=%d H=%d W=%d)", layers, B, H, W);
    if ((reinterpret_cast<uintptr_t>(scratch) & 15) != 0)
        return dg::nn_fail(DG_EINVAL, "dg_nn_forward_tc: scratch must be 16-byte aligned");
    int64_t elems = 0, most = 0;
    for (int l = 0; l < layers; ++l) {
        if (!w[l] || !b[l]) return dg::nn_fail(DG_EINVAL, "dg_nn_forward_tc: null pointer");
        n.w[l] = w[l];
        n.CI[l] = channels[l];
        n.CO[l] = channels[l + 1];
        n.NT[l] = dg::nt_of(channels[l + 1]);
        const int64_t e = dg::wimg_elems(n.CI[l], n.CO[l], n.NT[l]);
        elems = n.off[l] + (e + 7) / 8 * 8;
        most = std::max(most, e / 8);
    }
    cudaStream_t s = (cudaStream_t)stream;
    uint16_t *wimg = reinterpret_cast<uint16_t *>(scratch);
    const bool b16 = dg::net16(channels, layers);
    float *buf[2] = {scratch + elems / 2, scratch + elems / 2 + act};
    // both buffers' planes follow one another
    const int64_t planes = b16 ? act / 4 * (layers > 2 ? 2 : 1) / ((int64_t)(H + 2) * (W + 2)) : 0;
    if (b16) most = std::max(most, planes * 2 * ((int64_t)W + 2 + H));
    dg::k_net_tc_wimg<<<dim3((unsigned)std::min<int64_t>((most + 255) / 256, 152 * 2), (unsigned)(layers + (b16 ? 1 : 0))), 256, 0, s>>>(
        n, wimg, layers, reinterpret_cast<uint4 *>(buf[0]), planes, H, W);
    cudaError_t e = cudaGetLastError();
    const float *h = x;
    for (int l = 0; l < layers && e == cudaSuccess; ++l) {
        float *z = l + 1 == layers ? y : buf[l & 1];
        e = dg::launch_conv_blocks(h, wimg + n.off[l], b[l], z, B, channels[l], channels[l + 1], H, W, s, l + 1 < layers,
                                   b16 && l > 0, b16 && l + 1 < layers);
        h = z;
    }
    return dg::nn_done(e, "dg_nn_forward_tc");
}

int64_t dg_nn_conv3x3_tc_scratch(int32_t B, int32_t Ci, int32_t Co, int32_t H, int32_t W)
{
    if (!dg::tc_shape_ok(B, Ci, Co, H, W)) return -1;
    if (Co > 128) return dg::fwd_scratch(Ci, Co);  // the backward refuses this shape
    return dg::nn_conv_tc_scratch(B, Ci, Co, H, W);
}

dg_status dg_nn_conv3x3_backward_tc(const float *x, const float *w, const float *dy, float *dx, float *dw, float *db,
                                    int32_t B, int32_t Ci, int32_t Co, int32_t H, int32_t W, float *scratch,
                                    void *stream)
{
    if (!x || !w || !dy || !dw || !db || !scratch)
        return dg::nn_fail(DG_EINVAL, "dg_nn_conv3x3_backward_tc: null pointer");
    if (!dg::tc_shape_ok(B, Ci, Co, H, W))
        return dg::nn_fail(DG_EINVAL, "dg_nn_conv3x3_backward_tc: bad shape B=%d Ci=%d Co=%d H=%d W=%d", B, Ci, Co, H, W);
    if (Co > 128)
        return dg::nn_fail(DG_EUNSUPPORTED, "dg_nn_conv3x3_backward_tc: at most 128 output channels (Co=%d)", Co);
    if ((reinterpret_cast<uintptr_t>(scratch) & 15) != 0)
        return dg::nn_fail(DG_EINVAL, "dg_nn_conv3x3_backward_tc: scratch must be 16-byte aligned");
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaSuccess;
    if (dx) e = dg::launch_conv_tc(true, dy, w, nullptr, dx, B, Co, Ci, H, W, reinterpret_cast<uint16_t *>(scratch), s);
    float *part = scratch + dg::bwd_wimg_floats(Ci, Co);
    if (e != cudaSuccess) return dg::nn_done(e, "dg_nn_conv3x3_backward_tc");
    unsigned *err = dg::err_word();
    if (!err) return dg::nn_done(cudaErrorInvalidSymbol, "dg_nn_conv3x3_backward_tc");
    const dg::DwShape d = dg::dw_shape(B, Ci, H, W);
    const int smem = dg::dw_smem(d.tw);
    if ((e = cudaFuncSetAttribute(dg::k_conv3x3_dw_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess)
        return dg::nn_done(e, "dg_nn_conv3x3_backward_tc");
    const dim3 grid((unsigned)((Ci + dg::kDwCB - 1) / dg::kDwCB), (unsigned)d.S);
    dg::k_conv3x3_dw_tc<<<grid, dg::kDwThreads + 32, smem, s>>>(x, dy, part, Ci, Co, H, W, d.tw, d.nb, d.rows,
                                                                (d.rows + d.S - 1) / d.S, (int)d.S, err);
    if ((e = cudaGetLastError()) != cudaSuccess) return dg::nn_done(e, "dg_nn_conv3x3_backward_tc");
    const int64_t n = (int64_t)Co * (Ci * 9 + 1);
    dg::k_conv3x3_dw_tc_sum<<<(unsigned)std::min<int64_t>((n + 127) / 128, 152 * 16), 128, 0, s>>>(part, dw, db, Ci, Co,
                                                                                                   (int)d.S);
    return dg::nn_done(cudaGetLastError(), "dg_nn_conv3x3_backward_tc");
}

dg_status dg_nn_tc_check(void *stream)
{
    unsigned *err = dg::err_word();
    if (!err) return dg::nn_fail(DG_ECUDA, "dg_nn_tc_check: the error word has no device address");
    unsigned h = 0;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemcpyAsync(&h, err, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return dg::nn_done(e, "dg_nn_tc_check");
    if (h) {
        cudaMemsetAsync(err, 0, sizeof h, s);
        cudaStreamSynchronize(s);
        return dg::nn_fail(DG_ETIMEOUT, "a tensor-core layer's wait ran out; its outputs are not valid");
    }
    return DG_OK;
}

}  // extern "C"
