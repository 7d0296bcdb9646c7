// Learned k-predictor: a small convolutional network that estimates, from a
// 64 x 64 area-averaged copy of an image and a 16-bin histogram of its grey
// levels, how many passes (k) the method will take.  Not a method of the
// paper: its concluding section leaves choosing the iteration factor as
// future work.  The estimate only chooses a schedule; results and k are
// always those of the exact method.
//
// Network (weights from an offline fit on seeded synthetic images labelled
// with k by this library's exact denoiser; a sample of the labels is checked
// against the CPU oracle by the tests):
//   x0 = 64 x 64 x 1 area means / 255
//   x1..x4 = ReLU(conv3x3(x_{l-1}) + b_l), 16 channels, zero padding
//   g = mean of x4 over the 64 x 64 positions (16 values)
//   k_hat = max(0, w_h . [g, histogram] + b_h)
//
// The convolutions run on the 5th-generation tensor cores (tcgen05, BF16
// operands, FP32 accumulation in tensor memory) as implicit GEMMs with the 3 x
// 3 taps as K steps.  A 16-channel layer's input comes into shared memory by
// TMA as two planes of 8 channels, each a row-major list of 16-byte positions
// with a pitch of 66 and the zero border filled in by the copy.  In that
// layout 8 consecutive positions are one core matrix of the no-swizzle operand
// formats, K-major with the channels as K (the convolution) and MN-major with the
// positions as K (the weight gradients), and a tap is nothing but another start
// address: no operand is ever rearranged by threads.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/hgrms.h"
#include "kernels.h"

namespace hg {

namespace {

constexpr int kSide = 64;              // feature map side
constexpr int kPix = kSide * kSide;    // 4096 positions
constexpr int kCh = 16;                // channels
constexpr int kBins = 16;              // histogram bins
constexpr int kBlockM = 128;           // positions per CTA (MMA M)
constexpr int kBBytes = kCh * 16 * 2;         // one K step of B: 16 x 16 bf16

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor, no swizzle: start address, K-direction
// core-matrix stride (leading byte offset) and M/N-direction stride (stride
// byte offset), all in 16-byte units; descriptor version 1 (bit 46).
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo) { return (addr >> 4) | (lbo >> 4) << 16; }
__device__ __forceinline__ uint32_t desc_hi(uint32_t sbo) { return (sbo >> 4) | 1u << 14; }

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N = 16, M = 128.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kCh >> 3) << 17) |
                            ((uint32_t)(kBlockM >> 4) << 24);

// Byte offset of element (row, k) of a 16-wide K-major operand tile made of
// 8 x 8 core matrices: core matrix (row / 8, k / 8) at 256 (row / 8) +
// 128 (k / 8), rows of 16 bytes inside it.
__device__ __forceinline__ int core_off(int row, int k) {
    return (row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

__device__ __forceinline__ void mbar_init1(uint64_t* m, uint32_t count = 1) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(m)), "r"(count));
}
// Bounded wait for phase `parity` of an mbarrier.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* m, uint32_t parity) {
    for (uint32_t spins = 0; spins < (1u << 22); ++spins) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}"
            : "=r"(done)
            : "r"(smem_u32(m)), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
// The same; a wait that gives up records the error and waits once more, so
// that no copy or MMA of this CTA is left in flight when the CTA goes on.
__device__ __forceinline__ bool mbar_wait_or_flag(uint64_t* m, uint32_t parity, unsigned* err) {
    if (mbar_wait_bounded(m, parity)) return true;
    atomicExch(err, 1u);
    return mbar_wait_bounded(m, parity);
}
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t tmem, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols));
}
// One MMA, issued by the lane whose `lead` is set; operand descriptors as (low,
// high) words.  The low word holds the start address in 16-byte units, so
// stepping through an operand is an add to it.  The whole warp runs the loops
// around it with the same values: descriptors live in uniform registers, and
// code that only one thread reaches has to move every one of them there first.
__device__ __forceinline__ void mma_f16(uint32_t lead, uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                        uint32_t b_hi, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n.reg .b64 a, b;\n.reg .pred p, q;\nmov.b64 a, {%1, %2};\nmov.b64 b, {%3, %4};\nsetp.ne.u32 p, %6, 0;\n"
        "setp.ne.u32 q, %7, 0;\n@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}" ::"r"(d),
        "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc), "r"(lead)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t lead, uint64_t* m) {
    asm volatile(
        "{\n.reg .pred q;\nsetp.ne.u32 q, %1, 0;\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(smem_u32(m)),
        "r"(lead)
        : "memory");
}
// 1 in one lane of the (converged) warp.
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t lead;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(lead));
    return lead;
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// TMA load of one 8-channel plane of image `img`: rows from y, columns from x
// (positions outside the image read as zeros; the innermost coordinate is
// channel 0 or 8, a 16-byte boundary).
__device__ __forceinline__ void tma_plane(void* dst, const CUtensorMap* map, int half, int x, int y, int img,
                                          uint64_t* m) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_u32(dst)),
        "l"(map), "r"(8 * half), "r"(x), "r"(y), "r"(img), "r"(smem_u32(m))
        : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* m, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(m)), "r"(bytes) : "memory");
}

constexpr int kPitch = kSide + 2;  // positions per row with the border

// One channel of an image (64 x 64 bf16) with a border of zeros into s_x (66 x 66).
__device__ __forceinline__ void load_bordered(const __nv_bfloat16* __restrict__ x, float* s_x) {
    for (int i = threadIdx.x; i < kPitch * kPitch; i += blockDim.x) {
        const int y = i / kPitch - 1, xx = i % kPitch - 1;
        s_x[i] = y >= 0 && y < kSide && xx >= 0 && xx < kSide ? __bfloat162float(x[y * kSide + xx]) : 0.f;
    }
}

// The first layer: one input channel, 9 taps, 16 output channels.  in
// [image][64][64], out [image][64][64][16] bf16; w the parameters [tap][16] in
// fp32, rounded to bf16 here; bias 16 floats.  On the CUDA cores, products of
// bf16 values summed in fp32: as a tensor-core GEMM its K is 9 and its operand
// has to be gathered value by value, which took 30 us for 256 images.  CTA
// (image); a thread keeps the weights of 8 channels in registers and computes
// 32 positions.  256 images: 14 us (33.5 MB out).
__global__ void __launch_bounds__(256) conv1_kernel(const __nv_bfloat16* __restrict__ in, const float* __restrict__ w,
                                                    const float* __restrict__ bias, __nv_bfloat16* __restrict__ out) {
    __shared__ float s_x[kPitch * kPitch];
    const int tid = threadIdx.x, h = tid & 1;
    load_bordered(in + (size_t)blockIdx.x * kPix, s_x);
    float wr[9][8], br[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        br[c] = bias[8 * h + c];
#pragma unroll
        for (int t = 0; t < 9; ++t) wr[t][c] = __bfloat162float(__float2bfloat16_rn(w[t * kCh + 8 * h + c]));
    }
    __syncthreads();
    __nv_bfloat16* dst = out + (size_t)blockIdx.x * kPix * kCh + 8 * h;
    for (int p = tid >> 1; p < kPix; p += 128) {
        const float* sx = s_x + (p >> 6) * kPitch + (p & 63);
        float acc[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = br[c];
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const float x = sx[(t / 3) * kPitch + t % 3];
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] = fmaf(x, wr[t][c], acc[c]);
        }
        __align__(16) __nv_bfloat16 o[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) o[c] = __float2bfloat16_rn(fmaxf(acc[c], 0.f));
        *reinterpret_cast<uint4*>(dst + (size_t)p * kCh) = *reinterpret_cast<const uint4*>(o);
    }
}

// A 16-channel layer: out[p][co] = ReLU(bias[co] + sum over taps and ci of in[p +
// tap][ci] w[tap][ci][co]).  CTA (b, image) computes kBand rows: their input
// rows are kBand + 2 rows of the two channel planes, position (y, x) of the
// padded band at 66 y + x.  Output q = 66 y + x (x < 64 is a pixel, the other
// two are padding and are dropped) takes tap (ky, kx) from input q + 66 ky + kx,
// so the A operand of a tap is the plane pair from that position on: 128
// positions per MMA (M), two core matrices of 8 channels (K = 16, a plane
// apart), 5 MMA tiles of 9 taps with an accumulator of 16 columns each.
//
// With mask != null the kernel computes the gradient of a layer's input
// instead (back-propagation through a 16-channel convolution): `in` is the
// gradient of the layer's output, the taps' offsets are negated, w holds the
// transposed weights (output channel = the layer's input channel), and the
// result is multiplied by (mask > 0), the ReLU of the layer's input.
//
// Bound by the operand reads of the MMAs from shared memory (4 KB each, about
// 70 cycles; N is only 16).  8 rows a CTA leave four CTAs per SM (their 128
// tensor-memory columns each are all there are), so loads, MMAs and epilogues
// of different CTAs overlap; 4 rows and eight CTAs per SM measured the same.
// 256 images: 27 us forward and backward (67 and 101 MB), 59 us when every
// thread gathered the 9 taps of its position.
constexpr int kBand = 8;
constexpr int kBandTiles = ((kBand - 1) * kPitch + kSide + kBlockM - 1) / kBlockM;  // 5
constexpr int kConvPlane = (kBandTiles * kBlockM + 2 * kPitch + 2 + 7) / 8 * 128;    // bytes; every position an MMA reads
constexpr int kConvCols = 128;
constexpr size_t kConvSmem = 50 * 1024;  // four CTAs per SM
static_assert(kBandTiles * kCh <= kConvCols, "accumulator columns");
static_assert(2 * kConvPlane + 9 * kBBytes + 128 <= (int)kConvSmem && (kBand + 2) * kPitch * 16 <= kConvPlane, "conv planes");

__global__ void __launch_bounds__(128) conv16_tc_kernel(const __grid_constant__ CUtensorMap in,
                                                        const uint8_t* __restrict__ w, const float* __restrict__ bias,
                                                        __nv_bfloat16* __restrict__ out, unsigned* __restrict__ err,
                                                        const __nv_bfloat16* __restrict__ mask) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t full, done[kBandTiles];
    __shared__ uint32_t tmem_base;
    __shared__ float s_bias[kCh];
    if (smem_u32(smem) & 127u) {  // TMA destinations need 128-byte boundaries
        if (threadIdx.x == 0) atomicExch(err, 1u);
        return;
    }
    uint8_t* sB = smem + 2 * kConvPlane;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int img = blockIdx.y, y0 = blockIdx.x * kBand;
    if (tid == 0) {
        mbar_init1(&full);
        for (int t = 0; t < kBandTiles; ++t) mbar_init1(&done[t]);
        asm volatile("fence.mbarrier_init.release.cluster;");
        asm volatile("fence.proxy.async.shared::cta;");
        mbar_expect(&full, 2u * (kBand + 2) * kPitch * 16);
        for (int h = 0; h < 2; ++h) tma_plane(smem + h * kConvPlane, &in, h, -1, y0 - 1, img, &full);
    }
    __syncwarp();
    if (warp == 0) tmem_alloc(&tmem_base, kConvCols);
    for (int i = tid; i < 9 * kBBytes / 16; i += 128)
        reinterpret_cast<uint4*>(sB)[i] = __ldg(reinterpret_cast<const uint4*>(w) + i);
    if (tid < kCh) s_bias[tid] = mask ? 0.f : bias[tid];
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_base;
    if (warp == 0) {
        const uint32_t lead = elect_one();
        mbar_wait_or_flag(&full, 0u, err);
        __syncwarp();
        // Tap (ky, kx) is 66 ky + kx positions from the tile's first one, or,
        // negated, as many back from position 134.
        const uint32_t a0 = desc_lo(smem_u32(smem), kConvPlane) + (mask ? 2u * kPitch + 2u : 0u);
        const uint32_t step = mask ? ~0u : 1u;
        const uint32_t b0 = desc_lo(smem_u32(sB), 128);
#pragma unroll
        for (int t = 0; t < kBandTiles; ++t) {
#pragma unroll
            for (int tap = 0; tap < 9; ++tap)
                mma_f16(lead, tmem + (uint32_t)(t * kCh),
                        a0 + (uint32_t)(t * kBlockM) + step * (uint32_t)((tap / 3) * kPitch + tap % 3), desc_hi(128),
                        b0 + (uint32_t)(tap * kBBytes / 16), desc_hi(256), kIdesc, tap > 0 ? 1u : 0u);
            mma_commit(lead, &done[t]);
        }
    }
    __syncwarp();
    // The mask values of this thread's positions, loaded while the MMAs run.
    uint4 mk[kBandTiles][2];
    if (mask) {
#pragma unroll
        for (int t = 0; t < kBandTiles; ++t) {
            const int q = t * kBlockM + 32 * warp + lane;
            const int y = q / kPitch, x = q - y * kPitch;
            if (x >= kSide || y >= kBand) continue;
            const uint4* mp = reinterpret_cast<const uint4*>(mask + ((size_t)img * kPix + (y0 + y) * kSide + x) * kCh);
            mk[t][0] = __ldg(mp);
            mk[t][1] = __ldg(mp + 1);
        }
    }
#pragma unroll
    for (int t = 0; t < kBandTiles; ++t) {
        const bool ok = __all_sync(0xffffffffu, mbar_wait_or_flag(&done[t], 0u, err));
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (!ok) continue;
        uint32_t r[16];
        tmem_ld16(tmem + (uint32_t)(t * kCh) + ((uint32_t)(32 * warp) << 16), r);
        const int q = t * kBlockM + 32 * warp + lane;
        const int y = q / kPitch, x = q - y * kPitch;
        if (x >= kSide || y >= kBand) continue;
        const size_t pos = (size_t)img * kPix + (y0 + y) * kSide + x;
        __align__(16) __nv_bfloat16 o[16];
        if (mask) {
            const uint32_t mw[8] = {mk[t][0].x, mk[t][0].y, mk[t][0].z, mk[t][0].w,
                                    mk[t][1].x, mk[t][1].y, mk[t][1].z, mk[t][1].w};
#pragma unroll
            for (int c = 0; c < 16; ++c) {  // bf16 is the high half of an fp32
                const float v = __uint_as_float(c & 1 ? mw[c / 2] & 0xFFFF0000u : mw[c / 2] << 16);
                o[c] = __float2bfloat16_rn(v > 0.f ? __uint_as_float(r[c]) : 0.f);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 16; ++c) o[c] = __float2bfloat16_rn(fmaxf(__uint_as_float(r[c]) + s_bias[c], 0.f));
        }
        uint4* dst = reinterpret_cast<uint4*>(out + pos * kCh);
        dst[0] = *reinterpret_cast<const uint4*>(&o[0]);
        dst[1] = *reinterpret_cast<const uint4*>(&o[8]);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        tmem_dealloc(tmem, kConvCols);
    }
}

// Features of image blockIdx.y: row i = blockIdx.x of the 64 x 64 area
// means (each cell averages rows [i R / 64, max((i+1) R / 64, i R / 64 + 1))
// and the matching columns) and that row band's share of the 16-bin
// histogram (bin = value / 16, counts / pixels, added into hist).
//
// Every byte is read once, for both.  A warp takes 512 columns (16 per lane, four
// 4-byte words realigned from five) of some rows of the band, three rows'
// loads at a time.  Column sums grow in 16-bit lanes (even and odd bytes) over
// up to 255 rows.  The histogram counts in registers: 16 counters of 4 bits, a
// shifted one per pixel, widened to 8 bits every 12 pixels and to the warp's
// totals every 240, so equal values in a warp - most of a smooth image - cost
// no conflicts.  Bound by its integer instructions.
// 64 images of 128..2048 pixels a side, 93 MB: 82 us (208 with an atomic on shared
// bins per pixel; 8 columns per lane 95, although fewer lanes idle at the
// images' right ends; 13.7 us to read the bytes).
constexpr int kFeatWarps = 4;

// Sixteen 4-bit counters (bin b: bits 4 b of hi:lo), widened to bytes: bins 0, 2, 4, 6 / 1, 3, 5, 7 / 8, ... / 9, ...
struct BinCounts {
    uint32_t lo = 0u, hi = 0u;
    uint32_t b[4] = {0u, 0u, 0u, 0u};
    // Two pixels: bytes j and j + 1 of s = 4 (value / 16) and of t = s ^ 32.  PTX
    // shifts by 32 and more give 0, so each pixel counts in lo or in hi.
    __device__ __forceinline__ void add2(uint32_t s, uint32_t t, int j) {
        lo += shl1(__byte_perm(s, 0u, 0x4440u + j)) + shl1(__byte_perm(s, 0u, 0x4441u + j));
        hi += shl1(__byte_perm(t, 0u, 0x4440u + j)) + shl1(__byte_perm(t, 0u, 0x4441u + j));
    }
    static __device__ __forceinline__ uint32_t shl1(uint32_t sh) {
        uint32_t r;
        asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(sh));
        return r;
    }
    __device__ __forceinline__ void widen() {  // before a 4-bit counter can reach 16
        b[0] += lo & 0x0F0F0F0Fu;
        b[1] += (lo >> 4) & 0x0F0F0F0Fu;
        b[2] += hi & 0x0F0F0F0Fu;
        b[3] += (hi >> 4) & 0x0F0F0F0Fu;
        lo = hi = 0u;
    }
    // Warp-collective, before a byte can reach 256 (widen first): the warp's totals into s[16].
    __device__ __forceinline__ void flush(unsigned* s, int lane) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t e = b[i] & 0x00FF00FFu, o = (b[i] >> 8) & 0x00FF00FFu;  // bytes 0, 2 and 1, 3
            e = __reduce_add_sync(0xffffffffu, e);
            o = __reduce_add_sync(0xffffffffu, o);
            // Byte j of b[i]: bin 8 (i / 2) + 2 j + (i & 1); lanes 4 i .. 4 i + 3 add one each.
            const int j = lane & 3;
            if (lane >> 2 == i) atomicAdd(&s[8 * (i >> 1) + (i & 1) + 2 * j], ((j & 1 ? o : e) >> (j & 2 ? 16 : 0)) & 0xFFFFu);
            b[i] = 0u;
        }
    }
};

__global__ void __launch_bounds__(kFeatWarps * 32) features_kernel(const ImgDesc* __restrict__ imgs,
                                                                   __nv_bfloat16* __restrict__ x0,
                                                                   float* __restrict__ hist, float* __restrict__ x0f) {
    const ImgDesc d = imgs[blockIdx.y];
    const int i = blockIdx.x, rows = d.rows, cols = d.cols;
    const int r0 = (int)((long long)i * rows / kSide);
    const int r1 = max(r0 + 1, (int)((long long)(i + 1) * rows / kSide));
    // Every row counts in one band's histogram; in images of fewer than 64
    // rows some bands repeat a row and count none.
    const bool count = (int)((long long)(i + 1) * rows / kSide) > r0;
    __shared__ unsigned s_hist[kBins];
    __shared__ unsigned s_cell[kSide];  // sums: at most 1024 x 1024 x 255
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid < kBins) s_hist[tid] = 0u;
    if (tid < kSide) s_cell[tid] = 0u;
    __syncthreads();
    const uint8_t* base = d.user;
    const bool wide = cols >= kSide;  // every column belongs to one cell
    // Warps: column blocks of 512, and where there are fewer than warps, every
    // split-th row of the band.
    const int blocks = (cols + 511) / 512;
    const int split = blocks == 1 ? kFeatWarps : (blocks == 2 ? kFeatWarps / 2 : 1);
    BinCounts bins;
    int groups = 0;          // of three rows since the last flush (warp-uniform)
    unsigned counted = 0u;   // pixels this warp put in the histogram, those outside the image (as zeros) too
    for (int t = warp; t < blocks * split; t += kFeatWarps) {
        const int part = t % split, x = (t / split) * 512 + 16 * lane;
        const int nx = min(16, cols - x);  // columns of this lane in the image (may be negative)
        uint32_t ok[4];  // their bytes
#pragma unroll
        for (int v = 0; v < 4; ++v) ok[v] = nx >= 4 * v + 4 ? ~0u : (nx > 4 * v ? (1u << (8 * (nx - 4 * v))) - 1u : 0u);
        for (int ra = r0 + part; ra < r1; ra += 255 * split) {
            const int rb = min(r1, ra + 255 * split);
            uint32_t even[4] = {0u, 0u, 0u, 0u}, odd[4] = {0u, 0u, 0u, 0u};
            for (int r = ra; r < rb; r += 3 * split) {
                // Three rows' loads first, so that they are in flight together:
                // the aligned words that hold bytes of these columns.
                // Everything else reads as 0, in all lanes alike.
                uint32_t w[3][4];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const int rr = r + k * split;
                    const uintptr_t ad = reinterpret_cast<uintptr_t>(base + (long long)rr * cols + x);
                    const uint32_t* q = reinterpret_cast<const uint32_t*>(ad & ~uintptr_t(3));
                    const int sb = (int)(ad & 3u), last = rr < rb ? sb + nx : 0;  // word i: bytes 4 i .. of [sb, last)
                    uint32_t u[5];
#pragma unroll
                    for (int i = 0; i < 5; ++i) u[i] = 4 * i < last ? __ldg(q + i) : 0u;
#pragma unroll
                    for (int v = 0; v < 4; ++v) w[k][v] = __funnelshift_r(u[v], u[v + 1], 8u * sb) & ok[v];
                }
#pragma unroll
                for (int k = 0; k < 3; ++k)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        even[v] += w[k][v] & 0x00FF00FFu;
                        odd[v] += (w[k][v] >> 8) & 0x00FF00FFu;
                    }
                if (!count) continue;
#pragma unroll
                for (int k = 0; k < 12; ++k) {
                    const uint32_t s4 = (w[k / 4][k % 4] >> 2) & 0x3C3C3C3Cu, t4 = s4 ^ 0x20202020u;
                    bins.add2(s4, t4, 0);
                    bins.add2(s4, t4, 2);
                    if (k % 3 == 2) bins.widen();  // every 12 pixels
                }
                counted += 3u * 512u;
                if (++groups == 5) {  // at most 240 pixels per byte counter
                    bins.flush(s_hist, lane);
                    groups = 0;
                }
            }
            // The column sums go to their cells: the first column's is the last j
            // with j cols / 64 < x + 1, the next begins at (j + 1) cols / 64.
            if (wide && nx > 0) {
                int j = (kSide * (x + 1) - 1) / cols;
                int end = ((j + 1) * cols) >> 6;
                unsigned sum = 0u;
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const uint32_t v = c & 1 ? odd[c / 4] : even[c / 4];
                    if (x + c == end) {
                        atomicAdd(&s_cell[j], sum);
                        sum = 0u;
                        ++j;
                        end = ((j + 1) * cols) >> 6;
                    }
                    sum += c & 2 ? v >> 16 : v & 0xFFFFu;
                    if (c + 1 == nx) break;
                }
                atomicAdd(&s_cell[j], sum);
            }
        }
    }
    bins.flush(s_hist, lane);
    // Take the zeros from outside the image back out of bin 0.
    if (lane == 0 && counted) atomicAdd(&s_hist[0], 0u - counted);
    if (tid == 0 && count) atomicAdd(&s_hist[0], (unsigned)(r1 - r0) * (unsigned)cols);
    if (!wide) {
        // Narrow images: cells repeat columns.
        for (int j = tid; j < kSide; j += kFeatWarps * 32) {
            const int c0 = j * cols / kSide, c1 = max(c0 + 1, (j + 1) * cols / kSide);
            unsigned sum = 0u;
            for (int r = r0; r < r1; ++r)
                for (int c = c0; c < c1; ++c) sum += base[(long long)r * cols + c];
            s_cell[j] = sum;
        }
    }
    __syncthreads();
    if (tid < kSide) {
        const int c0 = (int)((long long)tid * cols / kSide);
        const int c1 = max(c0 + 1, (int)((long long)(tid + 1) * cols / kSide));
        const float mean = (float)s_cell[tid] / ((float)(r1 - r0) * (float)(c1 - c0) * 255.f);
        const size_t o = (size_t)blockIdx.y * kPix + (size_t)i * kSide + tid;
        x0[o] = __float2bfloat16_rn(mean);
        if (x0f) x0f[o] = mean;
    }
    if (tid < kBins && s_hist[tid])
        atomicAdd(&hist[blockIdx.y * kBins + tid], (float)s_hist[tid] / ((float)rows * (float)cols));
}

constexpr int kHeadThreads = 1024;  // one CTA per image: many loads in flight

// acc[c] += this thread's share of the sum over the positions of a layer's
// channel c (two 16-byte loads per position).
__device__ __forceinline__ void add_positions(const __nv_bfloat16* __restrict__ x, float (&acc)[kCh]) {
#pragma unroll 4
    for (int p = threadIdx.x; p < kPix; p += blockDim.x) {
        const uint4* q = reinterpret_cast<const uint4*>(x + (size_t)p * kCh);
        const uint4 a = __ldg(q), b = __ldg(q + 1);
        const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {  // bf16 is the high half of an fp32
            acc[2 * i] += __uint_as_float(w[i] << 16);
            acc[2 * i + 1] += __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
}

// k_hat of image blockIdx.x: mean of the last layer over the positions,
// then the linear head on [means, histogram].
__global__ void __launch_bounds__(kHeadThreads) head_kernel(const __nv_bfloat16* __restrict__ x4, const float* __restrict__ hist,
                                                   const float* __restrict__ wh, float* __restrict__ k_hat,
                                                   float* __restrict__ gap_out) {
    __shared__ float s_sum[kCh];
    if (threadIdx.x < kCh) s_sum[threadIdx.x] = 0.f;
    __syncthreads();
    float acc[kCh];
#pragma unroll
    for (int c = 0; c < kCh; ++c) acc[c] = 0.f;
    add_positions(x4 + (size_t)blockIdx.x * kPix * kCh, acc);
#pragma unroll
    for (int c = 0; c < kCh; ++c) {
        float v = acc[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum[c], v);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float y = wh[2 * kCh];  // bias
        for (int c = 0; c < kCh; ++c) {
            const float g = s_sum[c] / (float)kPix;
            if (gap_out) gap_out[blockIdx.x * kCh + c] = g;
            y += wh[c] * g + wh[kCh + c] * hist[blockIdx.x * kBins + c];
        }
        k_hat[blockIdx.x] = fmaxf(y, 0.f);
    }
}

// Weight and bias gradients of a 16-channel layer (back-propagation):
//   dW[tap][ci][co] += sum over positions p of X[p + off(tap)][ci] dY[p][co]
//   db[co]          += sum over p of dY[p][co]
// as GEMMs with the positions as K.  A task is kWBand rows of one image: the
// planes of X with their border and of dY with the same pitch (its two padding
// columns are zeros from outside the image, so what X holds there does not
// count).  Both operands are read MN-major as they lie: a core matrix is 8
// positions (K) of 8 channels (M or N).  A of (ky, 8 channels) has 8 such
// groups at a stride of one position: kx = 0, 1, 2 and five that are not used
// (M = 64 is the smallest; the strides of a plane and of a row do not fit one
// descriptor).  Six accumulators of 16 columns, and one with a matrix of
// ones as A for db, stay in tensor memory over all tasks of a CTA, one CTA per
// SM (so an FP32 sum runs over the bands of several images, 1024 positions each,
// before an atomic adds it to the others'; it ran over one image); the next
// task's planes load while this one's MMAs run.  One warp
// issues everything.  Bound by the operand reads from shared memory (2 KB per
// MMA, 7 x 66 MMAs a task, 35 cycles each).  256 images: 58 us; transposing both
// operands value by value, one 64-position chunk after another, took 190 us.
constexpr int kWBand = 16;
constexpr int kWSteps = kWBand * kPitch / 16;                                // K steps of 16 positions
constexpr int kXPlane = ((kWBand * kPitch + 2 * kPitch + 16) * 16 + 127) / 128 * 128;  // every position an MMA reads
constexpr int kYPlane = kWBand * kPitch * 16;
constexpr int kWStage = 2 * (kXPlane + kYPlane);
constexpr int kOnesBytes = 64 * 16 * 2;
constexpr size_t kWgradSmem = 2 * kWStage + kOnesBytes;
constexpr int kWCols = 128;
static_assert(kWBand * kPitch % 16 == 0 && kYPlane % 128 == 0 && kSide % kWBand == 0, "wgrad band");
// BF16, FP32 accumulation, both operands MN-major, N = 16, M = 64.
constexpr uint32_t kWgradIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                                 ((uint32_t)(kCh >> 3) << 17) | (4u << 24);

__global__ void __launch_bounds__(128) wgrad16_tc_kernel(const __grid_constant__ CUtensorMap xmap,
                                                         const __grid_constant__ CUtensorMap ymap, int images,
                                                         float* __restrict__ dW, float* __restrict__ db,
                                                         unsigned* __restrict__ err) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t full[2], freed[2];
    __shared__ uint32_t tmem_base;
    __shared__ int s_ok;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    constexpr int kTasks = kSide / kWBand;  // per image
    const int tasks = images * kTasks;
    uint8_t* ones = smem + 2 * kWStage;
    if (smem_u32(smem) & 127u) {  // TMA destinations need 128-byte boundaries
        if (tid == 0) atomicExch(err, 1u);
        return;
    }
    // Positions behind the loaded rows are read by MMAs (for padding columns,
    // against zeros of dY): they must be finite.
    for (int i = tid; i < 2 * kWStage / 16; i += 128) reinterpret_cast<uint4*>(smem)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = tid; i < kOnesBytes / 4; i += 128) reinterpret_cast<uint32_t*>(ones)[i] = 0x3F803F80u;
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init1(&full[i]);
            mbar_init1(&freed[i]);
        }
        asm volatile("fence.mbarrier_init.release.cluster;");
        s_ok = 1;
    }
    if (warp == 0) tmem_alloc(&tmem_base, kWCols);
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_base;
    if (warp == 0) {
        const uint32_t lead = elect_one();
        auto load = [&](int task, int st) {
            if (!lead) return;
            const int img = task / kTasks, y0 = (task % kTasks) * kWBand;
            uint8_t* p = smem + st * kWStage;
            mbar_expect(&full[st], 2u * ((kWBand + 2) * kPitch + kWBand * kPitch) * 16);
            for (int h = 0; h < 2; ++h) tma_plane(p + h * kXPlane, &xmap, h, -1, y0 - 1, img, &full[st]);
            for (int h = 0; h < 2; ++h) tma_plane(p + 2 * kXPlane + h * kYPlane, &ymap, h, 0, y0, img, &full[st]);
        };
        bool ok = true;
        int n = 0;  // tasks of this CTA so far
        int loads = 0;
        if ((int)blockIdx.x < tasks) {
            load(blockIdx.x, 0);
            ++loads;
        }
        for (int task = blockIdx.x; task < tasks && ok; task += gridDim.x, ++n) {
            const int st = n & 1;
            const uint32_t use = (uint32_t)(n >> 1);  // earlier uses of this stage
            const int next = task + gridDim.x;
            if (next < tasks) {
                // The other stage's MMAs (of task n - 1) must be done.
                if (n >= 1) ok = __all_sync(0xffffffffu, mbar_wait_or_flag(&freed[st ^ 1], (uint32_t)((n - 1) >> 1) & 1u, err));
                if (ok) {
                    load(next, st ^ 1);
                    ++loads;
                }
                __syncwarp();
            }
            ok = mbar_wait_or_flag(&full[st], use & 1u, err) && ok;
            ok = __all_sync(0xffffffffu, ok);
            const uint32_t x0 = smem_u32(smem + st * kWStage);
            uint32_t xd = desc_lo(x0, 128), yd = desc_lo(x0 + 2 * kXPlane, 128);
            const uint32_t od = desc_lo(smem_u32(ones), 1024);
            auto step = [&](uint32_t acc) {
#pragma unroll
                for (int j = 0; j < 6; ++j)  // (ky, half)
                    mma_f16(lead, tmem + 16u * j, xd + (uint32_t)((j & 1) * (kXPlane / 16) + (j >> 1) * kPitch), desc_hi(16), yd,
                            desc_hi(kYPlane), kWgradIdesc, acc);
                mma_f16(lead, tmem + 16u * 6, od, desc_hi(128), yd, desc_hi(kYPlane), kWgradIdesc, acc);
                xd += 16u;  // 16 positions
                yd += 16u;
            };
            step(n > 0 ? 1u : 0u);
#pragma unroll 2
            for (int k = 1; k < kWSteps; ++k) step(1u);
            mma_commit(lead, &freed[st]);
        }
        // A load that no task waited for (after a wait that gave up), and the last two tasks' MMAs.
        if (loads > n) mbar_wait_or_flag(&full[n & 1], (uint32_t)(n >> 1) & 1u, err);
        for (int b = n - 2 > 0 ? n - 2 : 0; b < n; ++b) ok = mbar_wait_or_flag(&freed[b & 1], (uint32_t)(b >> 1) & 1u, err) && ok;
        if (lead && (!ok || n == 0)) s_ok = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (s_ok) {
        // M = 64: rows 16 w .. 16 w + 15 in the first 16 lanes of warp w.
        const int row = 16 * warp + lane;
        for (int j = 0; j < 7; ++j) {
            uint32_t r[16];
            tmem_ld16(tmem + 16u * j + ((uint32_t)(32 * warp) << 16), r);
            if (lane >= 16) continue;
            if (j < 6 && row < 24) {
                const int tap = (j >> 1) * 3 + (row >> 3), ci = (j & 1) * 8 + (row & 7);
#pragma unroll
                for (int c = 0; c < kCh; ++c) atomicAdd(&dW[(tap * kCh + ci) * kCh + c], __uint_as_float(r[c]));
            }
            if (j == 6 && row == 0) {
#pragma unroll
                for (int c = 0; c < kCh; ++c) atomicAdd(&db[c], __uint_as_float(r[c]));
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        tmem_dealloc(tmem, kWCols);
    }
}

// The same for the first layer (one input channel): 9 x 16 sums per image,
// on the CUDA cores (a tensor-core tile of 9 useful rows of 64 would be mostly
// padding).  CTA (image); a thread takes 8 output channels of 32 positions
// and keeps its 9 x 8 sums in registers; products of bf16 values in fp32.
// 256 images: 27 us (33.5 MB of dY in); 125 us as a tensor-core GEMM.
__global__ void __launch_bounds__(256) wgrad1_kernel(const __nv_bfloat16* __restrict__ X,
                                                     const __nv_bfloat16* __restrict__ dY, float* __restrict__ dW,
                                                     float* __restrict__ db) {
    __shared__ float s_x[kPitch * kPitch];
    __shared__ float s_sum[10][kCh];
    const int tid = threadIdx.x, lane = tid & 31, h = tid & 1;
    load_bordered(X + (size_t)blockIdx.x * kPix, s_x);
    if (tid < 10 * kCh) s_sum[tid / kCh][tid % kCh] = 0.f;
    __syncthreads();
    float acc[10][8];
#pragma unroll
    for (int t = 0; t < 10; ++t)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[t][c] = 0.f;
    const __nv_bfloat16* src = dY + (size_t)blockIdx.x * kPix * kCh + 8 * h;
#pragma unroll 2
    for (int p = tid >> 1; p < kPix; p += 128) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(src + (size_t)p * kCh));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        float g[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // bf16 is the high half of an fp32
            g[2 * i] = __uint_as_float(w[i] << 16);
            g[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
        const float* sx = s_x + (p >> 6) * kPitch + (p & 63);
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const float x = sx[(t / 3) * kPitch + t % 3];
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[t][c] = fmaf(x, g[c], acc[t][c]);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[9][c] += g[c];
    }
#pragma unroll
    for (int t = 0; t < 10; ++t)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            float v = acc[t][c];
#pragma unroll
            for (int o = 16; o > 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane < 2) atomicAdd(&s_sum[t][8 * h + c], v);
        }
    __syncthreads();
    if (tid < 9 * kCh)
        atomicAdd(&dW[tid], s_sum[tid / kCh][tid % kCh]);
    else if (tid < 10 * kCh)
        atomicAdd(&db[tid - 9 * kCh], s_sum[9][tid - 9 * kCh]);
}

// Training head of image blockIdx.x: y = w . [means of x4, hist] + b (no
// ReLU while fitting), loss term (y - k)^2 / n, its gradient g = 2 (y - k) / n
// added into the head's gradients, and dgap[c] = g w[c] / 4096 for the
// backward pass.
__global__ void __launch_bounds__(kHeadThreads) train_head_kernel(const __nv_bfloat16* __restrict__ x4,
                                                         const float* __restrict__ hist, const float* __restrict__ k,
                                                         const float* __restrict__ wh, int n, float* __restrict__ gwh,
                                                         float* __restrict__ dgap, float* __restrict__ loss) {
    __shared__ float s_sum[kCh];
    if (threadIdx.x < kCh) s_sum[threadIdx.x] = 0.f;
    __syncthreads();
    float acc[kCh];
#pragma unroll
    for (int c = 0; c < kCh; ++c) acc[c] = 0.f;
    add_positions(x4 + (size_t)blockIdx.x * kPix * kCh, acc);
#pragma unroll
    for (int c = 0; c < kCh; ++c) {
        float v = acc[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum[c], v);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const float* hb = hist + blockIdx.x * kBins;
        float y = wh[2 * kCh];
        for (int c = 0; c < kCh; ++c) y += wh[c] * (s_sum[c] / (float)kPix) + wh[kCh + c] * hb[c];
        const float e = y - k[blockIdx.x];
        atomicAdd(loss, e * e / (float)n);
        const float g = 2.f * e / (float)n;
        for (int c = 0; c < kCh; ++c) {
            atomicAdd(&gwh[c], g * (s_sum[c] / (float)kPix));
            atomicAdd(&gwh[kCh + c], g * hb[c]);
            dgap[blockIdx.x * kCh + c] = g * wh[c] / (float)kPix;
        }
        atomicAdd(&gwh[2 * kCh], g);
    }
}

// Gradient of the last layer's output: dgap broadcast over the positions,
// times the ReLU of that output.
// One thread takes 8 channels of a position (16 bytes); 256 images 10 us (67
// MB), 163 us value by value.
__global__ void __launch_bounds__(256) train_dx4_kernel(const __nv_bfloat16* __restrict__ x4,
                                                        const float* __restrict__ dgap, int n,
                                                        __nv_bfloat16* __restrict__ dx4) {
    const int total = n * kPix * 2;  // n <= 4096
    for (int i = blockIdx.x * 256 + threadIdx.x; i < total; i += gridDim.x * 256) {
        const int img = i / (kPix * 2), h = i & 1;
        __align__(16) __nv_bfloat16 v[8], o[8];
        *reinterpret_cast<uint4*>(v) = __ldg(reinterpret_cast<const uint4*>(x4) + i);
        const float4* g = reinterpret_cast<const float4*>(dgap + img * kCh + 8 * h);
        const float4 g0 = __ldg(g), g1 = __ldg(g + 1);
        const float gv[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
        for (int c = 0; c < 8; ++c) o[c] = __float2bfloat16_rn(__bfloat162float(v[c]) > 0.f ? gv[c] : 0.f);
        reinterpret_cast<uint4*>(dx4)[i] = *reinterpret_cast<const uint4*>(o);
    }
}

// Adam step on the parameter vector (gradients g): m, v moments, step t.
__global__ void adam_kernel(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float b1, float b2, float eps, int t) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / (1.f - powf(b1, (float)t));
    const float vh = vi / (1.f - powf(b2, (float)t));
    w[i] -= lr * mh / (sqrtf(vh) + eps);
}

// x0 (bf16) of the selected images: out[b] = in[idx[b]].
__global__ void gather_kernel(const __nv_bfloat16* __restrict__ in, const float* __restrict__ hist_in,
                              const float* __restrict__ k_in, const int* __restrict__ idx, int n,
                              __nv_bfloat16* __restrict__ out, float* __restrict__ hist_out, float* __restrict__ k_out) {
    const int b = blockIdx.x;
    if (b >= n) return;
    const int j = idx[b];
    for (int p = threadIdx.x; p < kPix; p += blockDim.x) out[(size_t)b * kPix + p] = in[(size_t)j * kPix + p];
    if (threadIdx.x < kBins) hist_out[b * kBins + threadIdx.x] = hist_in[j * kBins + threadIdx.x];
    if (threadIdx.x == 0) k_out[b] = k_in[j];
}

// Parameter vector (hgrms_predictor_load's order) -> the B operand images of
// layers 2..4 for the forward pass (element (n = output channel, k = input
// channel)) and for the backward pass through their input (element (n = input
// channel, k = output channel)), bf16, rounded to nearest even.
struct PackedLayers {
    uint8_t* fwd[3];
    uint8_t* bwd[3];  // null: not wanted
};
__global__ void pack_kernel(const float* __restrict__ wv, PackedLayers out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;  // over 6 x 9 steps x 256 elements
    if (i >= 6 * 9 * 256) return;
    const int which = i / (9 * 256), rem = i % (9 * 256), layer = which % 3;
    const int step = rem / 256, n = (rem % 256) / 16, k = rem % 16;
    const float* wl = wv + 144 + layer * 2304;
    uint8_t* dst = which < 3 ? out.fwd[layer] : out.bwd[layer];
    if (!dst) return;
    const float v = which < 3 ? wl[(step * kCh + k) * kCh + n] : wl[(step * kCh + n) * kCh + k];
    *reinterpret_cast<__nv_bfloat16*>(dst + step * kBBytes + core_off(n, k)) = __float2bfloat16_rn(v);
}

static cudaError_t launch_pack(const float* w, const PackedLayers& out, cudaStream_t s) {
    pack_kernel<<<(6 * 9 * 256 + 255) / 256, 256, 0, s>>>(w, out);
    return cudaGetLastError();
}

// fp32 -> bf16, nearest even.
__global__ void to_bf16_kernel(const float* __restrict__ in, long long n, __nv_bfloat16* __restrict__ out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = __float2bfloat16_rn(in[i]);
}

constexpr int kNW = 144 + 3 * 2304 + 64 + 33;  // parameters
constexpr int kBiasOff = 144 + 3 * 2304;
constexpr int kHeadOff = kBiasOff + 64;

}  // namespace

// Tensor map of a [n][64][64][16] bf16 layer for tma_plane: boxes of 8
// channels, 66 columns and `rows` rows of one image.
static bool layer_map(CUtensorMap* m, const __nv_bfloat16* base, int n, int rows) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)kCh, (cuuint64_t)kSide, (cuuint64_t)kSide, (cuuint64_t)n};
    const cuuint64_t strides[3] = {kCh * 2, kSide * kCh * 2, (cuuint64_t)kPix * kCh * 2};
    const cuuint32_t box[4] = {8, (cuuint32_t)kPitch, (cuuint32_t)rows, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static cudaError_t launch_conv1(const __nv_bfloat16* in, int n, const float* w, const float* bias, __nv_bfloat16* out,
                                cudaStream_t s) {
    conv1_kernel<<<(unsigned)n, 256, 0, s>>>(in, w, bias, out);
    return cudaGetLastError();
}
static cudaError_t launch_conv16(const CUtensorMap& in, int n, const uint8_t* w, const float* bias, __nv_bfloat16* out,
                                 unsigned* err, const __nv_bfloat16* mask, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(conv16_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kConvSmem);
    if (e != cudaSuccess) return e;
    conv16_tc_kernel<<<dim3(kSide / kBand, (unsigned)n), 128, kConvSmem, s>>>(in, w, bias, out, err, mask);
    return cudaGetLastError();
}
static cudaError_t launch_wgrad16(const CUtensorMap& x, const CUtensorMap& dy, int n, float* dW, float* db, unsigned* err,
                                  int sms, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(wgrad16_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWgradSmem);
    if (e != cudaSuccess) return e;
    const int tasks = n * (kSide / kWBand);
    wgrad16_tc_kernel<<<(unsigned)(tasks < sms ? tasks : sms), 128, kWgradSmem, s>>>(x, dy, n, dW, db, err);
    return cudaGetLastError();
}

// Device buffers of the predictor for up to `cap` images.
struct Predictor {
    float* w = nullptr;                                      // the parameters (kNW)
    uint8_t* packed[3] = {nullptr, nullptr, nullptr};        // B operand images of layers 2..4
    __nv_bfloat16* x0 = nullptr;                             // cap x 4096
    __nv_bfloat16* act[2] = {nullptr, nullptr};              // cap x 4096 x 16, ping-pong
    float* hist = nullptr;                                   // cap x 16
    float* khat = nullptr;                                   // cap
    unsigned* err = nullptr;
    CUtensorMap act_map[2];  // of act[0], act[1]
    int cap = 0;
    bool loaded = false;
};

Predictor* predictor_new() { return new Predictor(); }

void predictor_free(Predictor* p) {
    if (!p) return;
    for (int l = 0; l < 3; ++l) cudaFree(p->packed[l]);
    cudaFree(p->w);
    cudaFree(p->x0);
    cudaFree(p->act[0]);
    cudaFree(p->act[1]);
    cudaFree(p->hist);
    cudaFree(p->khat);
    cudaFree(p->err);
    delete p;
}

// weights: layer l (0..3) as [tap 0..8][cin][16] floats (cin = 1 for l = 0,
// else 16), then 4 x 16 biases, then the head: 16 weights on the channel
// means, 16 on the histogram, 1 bias.
int predictor_load(Predictor* p, const float* weights, int n) {
    if (n != kNW) return HGRMS_EINVAL;
    if (!p->w && cudaMalloc(&p->w, kNW * sizeof(float)) != cudaSuccess) return HGRMS_ENOMEM;
    PackedLayers pk = {};
    for (int l = 0; l < 3; ++l) {
        if (!p->packed[l] && cudaMalloc(&p->packed[l], 9 * kBBytes) != cudaSuccess) return HGRMS_ENOMEM;
        pk.fwd[l] = p->packed[l];
    }
    if (!p->err && cudaMalloc(&p->err, sizeof(unsigned)) != cudaSuccess) return HGRMS_ENOMEM;
    if (cudaMemcpy(p->w, weights, kNW * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return HGRMS_ECUDA;
    // Done before the call returns: later calls may run on another stream.
    if (launch_pack(p->w, pk, nullptr) != cudaSuccess || cudaStreamSynchronize(nullptr) != cudaSuccess) return HGRMS_ECUDA;
    p->loaded = true;
    return HGRMS_OK;
}

static int predictor_reserve(Predictor* p, int n) {
    if (n <= p->cap) return HGRMS_OK;
    cudaFree(p->x0);
    cudaFree(p->act[0]);
    cudaFree(p->act[1]);
    cudaFree(p->hist);
    cudaFree(p->khat);
    p->x0 = nullptr;
    p->act[0] = p->act[1] = nullptr;
    p->hist = p->khat = nullptr;
    p->cap = 0;
    if (cudaMalloc(&p->x0, (size_t)n * kPix * sizeof(__nv_bfloat16)) != cudaSuccess ||
        cudaMalloc(&p->act[0], (size_t)n * kPix * kCh * sizeof(__nv_bfloat16)) != cudaSuccess ||
        cudaMalloc(&p->act[1], (size_t)n * kPix * kCh * sizeof(__nv_bfloat16)) != cudaSuccess ||
        cudaMalloc(&p->hist, (size_t)n * kBins * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&p->khat, (size_t)n * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        return HGRMS_ENOMEM;
    }
    for (int i = 0; i < 2; ++i)
        if (!layer_map(&p->act_map[i], p->act[i], n, kBand + 2)) return HGRMS_ECUDA;
    p->cap = n;
    return HGRMS_OK;
}

// Features and network for n images described by the device table `imgs`
// (their `user` pointers: device-readable image bytes).  k_hat (host, n
// floats) receives the estimates; x0_host / gap_host (optional, host) the
// area means and the last layer's channel means, for tests.
int predictor_run(Predictor* p, const ImgDesc* imgs, int n, cudaStream_t s, float* k_hat, float* x0_host,
                  float* hist_host, float* gap_host) {
    if (!p->loaded) return HGRMS_EINVAL;
    if (n <= 0) return HGRMS_OK;
    int rc = predictor_reserve(p, n);
    if (rc < 0) return rc;
    float* x0f = nullptr;
    float* gap = nullptr;
    if (x0_host && cudaMalloc(&x0f, (size_t)n * kPix * sizeof(float)) != cudaSuccess) return HGRMS_ENOMEM;
    if (gap_host && cudaMalloc(&gap, (size_t)n * kCh * sizeof(float)) != cudaSuccess) {
        cudaFree(x0f);
        return HGRMS_ENOMEM;
    }
    cudaError_t e = cudaMemsetAsync(p->hist, 0, (size_t)n * kBins * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(p->err, 0, sizeof(unsigned), s);
    if (e == cudaSuccess) {
        features_kernel<<<dim3(kSide, (unsigned)n), kFeatWarps * 32, 0, s>>>(imgs, p->x0, p->hist, x0f);
        e = cudaGetLastError();
    }
    const __nv_bfloat16* in = p->x0;
    for (int l = 0; l < 4 && e == cudaSuccess; ++l) {
        __nv_bfloat16* out = p->act[l & 1];
        const float* bias = p->w + kBiasOff + 16 * l;
        e = l == 0 ? launch_conv1(in, n, p->w, bias, out, s)
                   : launch_conv16(p->act_map[(l - 1) & 1], n, p->packed[l - 1], bias, out, p->err, nullptr, s);
        in = out;
    }
    if (e == cudaSuccess) {
        head_kernel<<<(unsigned)n, kHeadThreads, 0, s>>>(in, p->hist, p->w + kHeadOff, p->khat, gap);
        e = cudaGetLastError();
    }
    unsigned err = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(k_hat, p->khat, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&err, p->err, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && x0_host)
        e = cudaMemcpyAsync(x0_host, x0f, (size_t)n * kPix * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && hist_host)
        e = cudaMemcpyAsync(hist_host, p->hist, (size_t)n * kBins * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && gap_host)
        e = cudaMemcpyAsync(gap_host, gap, (size_t)n * kCh * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(x0f);
    cudaFree(gap);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? HGRMS_ENOMEM : HGRMS_ECUDA;
    return err ? HGRMS_ETIMEOUT : HGRMS_OK;
}

}  // namespace hg

namespace hg {

namespace {

// Device state of a fit, in one allocation.
struct Trainer {
    int n = 0, batch = 0;
    uint8_t* arena = nullptr;
    __nv_bfloat16* x0 = nullptr;  // n x 4096
    float* hist = nullptr;        // n x 16
    float* k = nullptr;           // n
    int* idx = nullptr;           // n: the epoch's permutation
    __nv_bfloat16* xb = nullptr;  // batch x 4096
    float* hb = nullptr;
    float* kb = nullptr;
    __nv_bfloat16* act[4] = {};   // batch x 4096 x 16
    __nv_bfloat16* grad[2] = {};  // batch x 4096 x 16
    float* dgap = nullptr;
    float* w = nullptr;           // parameters
    float* g = nullptr;           // gradients
    float* m = nullptr;
    float* v = nullptr;
    float* loss = nullptr;        // n / batch: the epoch's minibatches
    unsigned* err = nullptr;
    PackedLayers packed = {};
    // Tensor maps of act[0..2] and grad[0..1]: for the convolutions (input
    // bands) and the weight gradients (X and dY bands).
    CUtensorMap act_conv[3], act_x[3], grad_conv[2], grad_y[2];
    int sms = 0;

    ~Trainer() { cudaFree(arena); }
};

int trainer_init(Trainer& t, const float* x0, const float* hist, const float* k, int n, int batch,
                 const float* weights, cudaStream_t s) {
    t.n = n;
    t.batch = batch;
    const size_t act = (size_t)batch * kPix * kCh * sizeof(__nv_bfloat16);
    size_t total = 0;
    // Two rounds: the sizes, then the addresses (256-byte boundaries).
    auto place = [&](auto*& p, size_t bytes) {
        if (t.arena) p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(t.arena + total);
        total += (bytes + 255) / 256 * 256;
    };
    for (int round = 0; round < 2; ++round) {
        total = 0;
        place(t.x0, (size_t)n * kPix * 2);
        place(t.hist, (size_t)n * kBins * 4);
        place(t.k, (size_t)n * 4);
        place(t.idx, (size_t)n * 4);
        place(t.xb, (size_t)batch * kPix * 2);
        place(t.hb, (size_t)batch * kBins * 4);
        place(t.kb, (size_t)batch * 4);
        for (auto*& a : t.act) place(a, act);
        for (auto*& a : t.grad) place(a, act);
        place(t.dgap, (size_t)batch * kCh * 4);
        place(t.w, kNW * 4);
        place(t.g, kNW * 4);
        place(t.m, kNW * 4);
        place(t.v, kNW * 4);
        place(t.loss, (size_t)(n / batch) * 4);
        place(t.err, 4);
        for (auto*& a : t.packed.fwd) place(a, 9 * kBBytes);
        for (auto*& a : t.packed.bwd) place(a, 9 * kBBytes);
        if (round == 0 && cudaMalloc(&t.arena, total) != cudaSuccess) {
            cudaGetLastError();
            t.arena = nullptr;
            return HGRMS_ENOMEM;
        }
    }
    for (int i = 0; i < 3; ++i)
        if (!layer_map(&t.act_conv[i], t.act[i], batch, kBand + 2) || !layer_map(&t.act_x[i], t.act[i], batch, kWBand + 2))
            return HGRMS_ECUDA;
    for (int i = 0; i < 2; ++i)
        if (!layer_map(&t.grad_conv[i], t.grad[i], batch, kBand + 2) || !layer_map(&t.grad_y[i], t.grad[i], batch, kWBand))
            return HGRMS_ECUDA;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&t.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return HGRMS_ECUDA;
    cudaError_t e = cudaSuccess;
    // x0 as it is, through the activations' memory, and to bf16 on the device.
    const size_t chunk = (size_t)batch * kCh / 2;  // images that fit act[0] in fp32
    for (size_t i = 0; i < (size_t)n && e == cudaSuccess; i += chunk) {
        const size_t c = std::min(chunk, (size_t)n - i) * kPix;
        e = cudaMemcpyAsync(t.act[0], x0 + i * kPix, c * 4, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) break;
        to_bf16_kernel<<<(unsigned)t.sms * 8, 256, 0, s>>>(reinterpret_cast<const float*>(t.act[0]), (long long)c,
                                                          t.x0 + i * kPix);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(t.hist, hist, (size_t)n * kBins * 4, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(t.k, k, (size_t)n * 4, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(t.w, weights, kNW * 4, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(t.m, 0, kNW * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(t.v, 0, kNW * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(t.err, 0, 4, s);
    return e == cudaSuccess ? HGRMS_OK : HGRMS_ECUDA;
}

// Gradient of the mean squared k error over the images t.idx[b0 .. b0 + nb) into
// t.g (their loss is added to *loss): forward through the layers, then back
// through them.  Nothing waits for the host.
cudaError_t trainer_grad(Trainer& t, int b0, int nb, float* loss, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(t.g, 0, kNW * 4, s);
    if (e != cudaSuccess) return e;
    gather_kernel<<<nb, 256, 0, s>>>(t.x0, t.hist, t.k, t.idx + b0, nb, t.xb, t.hb, t.kb);
    const float* bias = t.w + kBiasOff;
    e = launch_conv1(t.xb, nb, t.w, bias, t.act[0], s);
    for (int l = 1; l < 4 && e == cudaSuccess; ++l)
        e = launch_conv16(t.act_conv[l - 1], nb, t.packed.fwd[l - 1], bias + 16 * l, t.act[l], t.err, nullptr, s);
    if (e != cudaSuccess) return e;
    train_head_kernel<<<nb, kHeadThreads, 0, s>>>(t.act[3], t.hb, t.kb, t.w + kHeadOff, nb, t.g + kHeadOff, t.dgap, loss);
    train_dx4_kernel<<<t.sms * 8, 256, 0, s>>>(t.act[3], t.dgap, nb, t.grad[0]);
    e = cudaGetLastError();
    int cur = 0;
    const int woff[4] = {0, 144, 144 + 2304, 144 + 2 * 2304};
    for (int l = 3; l >= 1 && e == cudaSuccess; --l) {
        e = launch_wgrad16(t.act_x[l - 1], t.grad_y[cur], nb, t.g + woff[l], t.g + kBiasOff + 16 * l, t.err, t.sms, s);
        if (e == cudaSuccess)
            e = launch_conv16(t.grad_conv[cur], nb, t.packed.bwd[l - 1], nullptr, t.grad[cur ^ 1], t.err, t.act[l - 1], s);
        cur ^= 1;
    }
    if (e != cudaSuccess) return e;
    wgrad1_kernel<<<nb, 256, 0, s>>>(t.xb, t.grad[cur], t.g, t.g + kBiasOff);
    return cudaGetLastError();
}

}  // namespace

int predictor_grad(const float* weights, const float* x0, const float* hist, const float* k, int n, float* grads,
                   float* loss, cudaStream_t s) {
    if (n < 1 || n > 4096) return HGRMS_EINVAL;
    Trainer t;
    int rc = trainer_init(t, x0, hist, k, n, n, weights, s);
    if (rc < 0) return rc;
    std::vector<int> idx((size_t)n);
    for (int i = 0; i < n; ++i) idx[i] = i;
    cudaError_t e = cudaMemcpyAsync(t.idx, idx.data(), (size_t)n * 4, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(t.loss, 0, 4, s);
    if (e == cudaSuccess) e = launch_pack(t.w, t.packed, s);
    if (e == cudaSuccess) e = trainer_grad(t, 0, n, t.loss, s);
    unsigned err = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(grads, t.g, kNW * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(loss, t.loss, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&err, t.err, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return HGRMS_ECUDA;
    return err ? HGRMS_ETIMEOUT : HGRMS_OK;
}

int predictor_train(float* weights, const float* x0, const float* hist, const float* k, int n, int epochs, int batch,
                    float lr, unsigned long long seed, float* loss_out, cudaStream_t s) {
    if (n < 1 || batch < 1 || batch > 4096 || epochs < 0 || !(lr > 0.f)) return HGRMS_EINVAL;
    if (batch > n) batch = n;
    Trainer t;
    int rc = trainer_init(t, x0, hist, k, n, batch, weights, s);
    if (rc < 0) return rc;
    std::vector<int> perm((size_t)n);
    for (int i = 0; i < n; ++i) perm[i] = i;
    unsigned long long st = seed * 6364136223846793005ull + 1442695040888963407ull;
    auto next = [&st]() {  // 64-bit LCG, high bits
        st = st * 6364136223846793005ull + 1442695040888963407ull;
        return (uint32_t)(st >> 33);
    };
    cudaError_t e = launch_pack(t.w, t.packed, s);
    int step = 0;
    const int batches = n / batch;
    // The steps are queued without waiting for any; an epoch's upload of its
    // permutation (pageable memory) waits for the epoch before it.
    for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
        for (int i = n - 1; i > 0; --i) std::swap(perm[i], perm[next() % (uint32_t)(i + 1)]);
        const float lr_ep = ep >= (3 * epochs) / 4 ? lr / 3.f : lr;
        e = cudaMemcpyAsync(t.idx, perm.data(), (size_t)n * 4, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(t.loss, 0, (size_t)batches * 4, s);
        for (int b = 0; b < batches && e == cudaSuccess; ++b) {
            e = trainer_grad(t, b * batch, batch, t.loss + b, s);
            if (e != cudaSuccess) break;
            ++step;
            adam_kernel<<<(kNW + 255) / 256, 256, 0, s>>>(t.w, t.g, t.m, t.v, kNW, lr_ep, 0.9f, 0.999f, 1e-8f, step);
            e = cudaGetLastError();
            if (e == cudaSuccess) e = launch_pack(t.w, t.packed, s);
        }
    }
    std::vector<float> losses((size_t)batches, 0.f);
    if (e == cudaSuccess && epochs > 0)
        e = cudaMemcpyAsync(losses.data(), t.loss, (size_t)batches * 4, cudaMemcpyDeviceToHost, s);
    unsigned err = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(weights, t.w, kNW * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&err, t.err, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return HGRMS_ECUDA;
    double last = 0.0;  // the last epoch's mean loss
    for (float l : losses) last += l;
    if (loss_out) *loss_out = (float)(last / batches);
    return err ? HGRMS_ETIMEOUT : HGRMS_OK;
}

}  // namespace hg
