// Unfused one-pass kernel (one thread per pixel, global loads) and the kernels
// that begin and end a call.
//
// The unfused kernel evaluates Algorithms 1 and 2 directly for each pixel:
// card by gathering over the window (equal to the paper's scattered
// increments, because the window and the |difference| < alpha test are
// symmetric), then flag / sum / replacement.  It is the straightforward GPU
// form of the method, kept as a second, independent device path and as the
// unfused point of comparison for the fused tile kernel.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace hg {

template <int B>
__global__ void __launch_bounds__(256) plain_kernel(PassArgs a) {
    __shared__ int s_np;
    __shared__ unsigned s_cur, s_aux;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    if (tid == 0) {
        s_np = launch_passes(a.ctrl, 1);
        s_cur = __ldcg(&a.ctrl->cur);
        s_aux = __ldcg(&a.ctrl->aux);
    }
    __syncthreads();
    if (s_np == 0) return;
    const uint8_t* src = a.canvas[s_cur];
    uint8_t* dst = a.canvas[s_aux];
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    bool changed = false;
    if (x < a.cols && y < a.rows) {
        const long long off = (long long)(kPadY + y) * a.pitch + kPadX + x;
        const uint8_t* s = src + off;
        const int ip = *s;
        int outv = ip;
        const bool interior = x >= B && x < a.cols - B && y >= B && y < a.rows - B;
        if (interior) {
            int card = 0;
#pragma unroll
            for (int dy = -B; dy <= B; ++dy)
#pragma unroll
                for (int dx = -B; dx <= B; ++dx) {
                    const int v = s[dy * a.pitch + dx];
                    card += (v < ip + a.alpha && v > ip - a.alpha) ? 1 : 0;
                }
            if (card <= 2) {
                int sum = 0, flag = 0;
#pragma unroll
                for (int dy = -B; dy <= B; ++dy)
#pragma unroll
                    for (int dx = -B; dx <= B; ++dx) {
                        const int v = s[dy * a.pitch + dx];
                        if (!(v < ip + a.alpha + 1 && v > ip - a.alpha)) {
                            sum += v * v;
                            ++flag;
                        }
                    }
                constexpr int kPixCount = (2 * B + 1) * (2 * B + 1);
                if (flag > kPixCount - 3) outv = (int)floorf(__fsqrt_rn((float)(sum / flag)));
            }
        }
        dst[off] = (uint8_t)outv;
        changed = outv != ip;
    }
    const int any = __syncthreads_or(changed);
    if (tid == 0) finish_launch(a.ctrl, any ? 1u : 0u, 1, gridDim.x * gridDim.y, s_aux, s_cur);
}

cudaError_t launch_plain(int beta, const PassArgs& a, cudaStream_t s) {
    const dim3 block(32, 8);
    const dim3 grid((a.cols + 31) / 32, (a.rows + 7) / 8);
    switch (beta) {
        case 1: plain_kernel<1><<<grid, block, 0, s>>>(a); break;
        case 2: plain_kernel<2><<<grid, block, 0, s>>>(a); break;
        case 3: plain_kernel<3><<<grid, block, 0, s>>>(a); break;
        case 4: plain_kernel<4><<<grid, block, 0, s>>>(a); break;
        case 5: plain_kernel<5><<<grid, block, 0, s>>>(a); break;
        case 6: plain_kernel<6><<<grid, block, 0, s>>>(a); break;
        case 7: plain_kernel<7><<<grid, block, 0, s>>>(a); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// Everything a call needs cleared, in one launch: the control block, the
// change bitmaps (n16 16-byte words), the barrier and, for a batch, the
// per-image counts (nk words).  (One kernel for the control block and a memset
// for each of the others cost a call two to three launches more, ~1.5 us
// each.)
__global__ void call_init_kernel(Ctrl* __restrict__ c, unsigned max_k, uint4* __restrict__ bm, long long n16,
                                 GridBar* __restrict__ bar, unsigned* __restrict__ counts, long long nk) {
    let_next_start();
    const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x, gt = (long long)gridDim.x * blockDim.x;
    if (g == 0) {
        Ctrl z = {};
        z.aux = 1;
        z.max_k = max_k;
        *c = z;
        if (bar) bar->ctr[0].v = bar->ctr[1].v = 0ull;
    }
    for (long long i = g; i < nk; i += gt) counts[i] = 0u;
    for (long long i = g; i < n16; i += gt) bm[i] = make_uint4(0u, 0u, 0u, 0u);
}

cudaError_t launch_call_init(Ctrl* c, unsigned max_k, uint32_t* bm, long long n16, GridBar* bar, unsigned* counts,
                             long long nk, int sms, cudaStream_t s) {
    long long blocks = (std::max(n16, nk) + 1023) / 1024;  // four words a thread
    blocks = std::min(std::max(blocks, 1ll), (long long)sms * 8);
    call_init_kernel<<<(unsigned)blocks, 256, 0, s>>>(c, max_k, reinterpret_cast<uint4*>(bm), n16, bar, counts, nk);
    return cudaGetLastError();
}

// Dense user image (row r at img + r*cols) -> canvas interior, in 16-byte
// row chunks; vector accesses when the user rows are 16-byte aligned.
__global__ void copy_in_kernel(const uint8_t* __restrict__ img, int rows, int cols,
                               uint8_t* __restrict__ canvas, long long pitch, int vec) {
    const long long chunks = (cols + 15) / 16;
    const long long total = chunks * rows;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long r = i / chunks;
        const int x = (int)(i - r * chunks) * 16;
        const uint8_t* s = img + r * cols + x;
        uint8_t* d = canvas + (kPadY + r) * pitch + kPadX + x;
        const int n = min(16, cols - x);
        if (vec && n == 16) {
            *reinterpret_cast<uint4*>(d) = __ldg(reinterpret_cast<const uint4*>(s));
        } else {
            for (int b = 0; b < n; ++b) d[b] = s[b];
        }
    }
}

static unsigned copy_grid(int rows, int cols, int sms) {
    const long long total = (long long)((cols + 15) / 16) * rows;
    long long blocks = (total + 255) / 256;
    const long long cap = (long long)sms * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return (unsigned)blocks;
}

cudaError_t launch_copy_in(const uint8_t* img, int rows, int cols, uint8_t* canvas, long long pitch,
                           int sms, cudaStream_t s) {
    const int vec = (cols % 16 == 0) && ((reinterpret_cast<uintptr_t>(img) & 15u) == 0);
    copy_in_kernel<<<copy_grid(rows, cols, sms), 256, 0, s>>>(img, rows, cols, canvas, pitch, vec);
    return cudaGetLastError();
}

// The end of a call: canvas `cur` -> the caller's dense images, and the
// control block (and a batch's per-image k) -> page-locked host memory, which
// saves the call a copy or two behind this launch.
//
// A warp takes a piece of an image row of up to kPieceVecs 16-byte words,
// aligned in the destination: words whose bytes lie at the same alignment in
// the canvas (16-byte aligned rows) are moved as they are, others are put
// together by funnel shifts from two aligned chunks, the second one the next
// lane's; the ends of the row go byte by byte.  Bound by memory: 8192 x 8192
// takes 28 us (134 MB, 4.7 TB/s; a whole row per warp took 17 us more: too many
// rows open at once).  128 images of 128..2048 pixels a side, 157 MB, 92 us
// (101 from five 4-byte loads a word, about 330 when every 4-byte word, or
// every byte of an odd row, was gathered by itself); 3839 x 2161 9 us.
constexpr int kPieceVecs = 128;

__host__ __device__ inline int row_pieces(int cols) {
    return cols < 16 * kPieceVecs ? 1 : (cols / 16 + kPieceVecs - 1) / kPieceVecs;
}

__device__ __forceinline__ void copy_rows(const uint8_t* __restrict__ canvas, long long pitch,
                                          uint8_t* __restrict__ user, int rows, int cols, int warp, int nwarps,
                                          int lane) {
    const int pieces = row_pieces(cols);
    const int total = rows * pieces;
    for (int t = warp; t < total; t += nwarps) {
        const int r = pieces == 1 ? t : t / pieces, pc = t - r * pieces;
        const uint8_t* src = canvas + r * pitch;
        uint8_t* dst = user + (long long)r * cols;
        const int head = min(cols, (int)(-reinterpret_cast<uintptr_t>(dst) & 15u));
        const int nvec = (cols - head) / 16;
        const int v1 = min(nvec, (pc + 1) * kPieceVecs);
        uint4* dv = reinterpret_cast<uint4*>(dst + head);
        if (head == 0) {
#pragma unroll 4
            for (int v = pc * kPieceVecs + lane; v < v1; v += 32) dv[v] = reinterpret_cast<const uint4*>(src)[v];
        } else {
            // Word v's bytes lie in the 16-byte chunks v and v + 1 of the
            // canvas row: a lane loads chunk v and has the next one from the
            // next lane (its last lane from the first of the next 32).
            constexpr int kIt = kPieceVecs / 32;
            const int v0 = pc * kPieceVecs + lane;
            const uint4* sv = reinterpret_cast<const uint4*>(src);
            uint4 c[kIt + 1];
#pragma unroll
            for (int i = 0; i <= kIt; ++i) {
                const int v = i < kIt ? v0 + 32 * i : (pc + 1) * kPieceVecs;
                c[i] = v <= v1 ? sv[v] : make_uint4(0u, 0u, 0u, 0u);
            }
            const uint32_t sh = (uint32_t)(head & 3) * 8u;
#pragma unroll
            for (int i = 0; i < kIt; ++i) {
                const uint4 x = lane == 0 ? c[i + 1] : c[i];
                const int from = (lane + 1) & 31;
                const uint32_t n0 = __shfl_sync(0xffffffffu, x.x, from), n1 = __shfl_sync(0xffffffffu, x.y, from);
                const uint32_t n2 = __shfl_sync(0xffffffffu, x.z, from), n3 = __shfl_sync(0xffffffffu, x.w, from);
                uint32_t w0, w1, w2, w3, w4;
                switch (head >> 2) {  // the same for the whole warp
                    case 0: w0 = c[i].x, w1 = c[i].y, w2 = c[i].z, w3 = c[i].w, w4 = n0; break;
                    case 1: w0 = c[i].y, w1 = c[i].z, w2 = c[i].w, w3 = n0, w4 = n1; break;
                    case 2: w0 = c[i].z, w1 = c[i].w, w2 = n0, w3 = n1, w4 = n2; break;
                    default: w0 = c[i].w, w1 = n0, w2 = n1, w3 = n2, w4 = n3; break;
                }
                if (v0 + 32 * i < v1)
                    dv[v0 + 32 * i] = make_uint4(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh),
                                                 __funnelshift_r(w2, w3, sh), __funnelshift_r(w3, w4, sh));
            }
        }
        if (pc == pieces - 1) {
            if (lane < head) dst[lane] = src[lane];
            const int e = head + 16 * nvec + lane;
            if (e < cols && lane < 16) dst[e] = src[e];
        }
    }
}

__global__ void __launch_bounds__(256) call_finish_kernel(FinishArgs a) {
    wait_for_previous();
    const Ctrl* c = a.ctrl;
    const int lane = threadIdx.x & 31, warp = (blockIdx.x * 256 + threadIdx.x) >> 5, nwarps = gridDim.x * 8;
    const uint8_t* canvas = a.arena[__ldcg(&c->cur)];
    if (a.imgs) {
        const ImgDesc d = load_desc(a.imgs, blockIdx.y);
        if (d.user && a.write)
            copy_rows(canvas + d.off + (long long)kPadY * d.pitch + kPadX, d.pitch, d.user, d.rows, d.cols, warp, nwarps,
                      lane);
    } else if (a.write) {
        copy_rows(canvas + (long long)kPadY * a.pitch + kPadX, a.pitch, a.user, a.rows, a.cols, warp, nwarps, lane);
    }
    if (blockIdx.x == 0 && blockIdx.y == 0 && a.host_ctrl) {
        const unsigned* cw = reinterpret_cast<const unsigned*>(c);
        unsigned* hw = reinterpret_cast<unsigned*>(a.host_ctrl);
        for (int i = threadIdx.x; i < (int)(sizeof(Ctrl) / 4); i += 256) hw[i] = __ldcg(cw + i);
        if (a.host_img_k)
            for (int i = threadIdx.x; i < a.nimg; i += 256) a.host_img_k[i] = __ldcg(a.img_k + i);
    }
}

cudaError_t launch_call_finish(const FinishArgs& a, int sms, cudaStream_t s) {
    // One image: up to eight CTAs per SM.  A batch: the CTAs of its largest
    // image, limited to sixteen per SM over all images.
    long long gx = 1;
    if (a.write) gx = ((long long)a.rows * row_pieces(a.cols) + 7) / 8;
    const unsigned gy = a.imgs ? (unsigned)a.nimg : 1u;
    const long long cap = a.imgs ? std::max(((long long)sms * 16 + gy - 1) / gy, 16ll) : (long long)sms * 8;
    gx = std::min(std::max(gx, 1ll), cap);
    return launch_dependent(call_finish_kernel, dim3((unsigned)gx, gy), dim3(256), 0, s, a);
}

// tile_img[b] = the image that fused tile b belongs to.
__global__ void tile_map_kernel(const ImgDesc* __restrict__ imgs, int nimg, int total_tiles, int* __restrict__ tile_img) {
    const int i = blockIdx.x;
    const int t0 = imgs[i].tile0;
    const int t1 = i + 1 < nimg ? imgs[i + 1].tile0 : total_tiles;
    for (int t = t0 + threadIdx.x; t < t1; t += blockDim.x) tile_img[t] = i;
}

__global__ void rms_kernel(const int* __restrict__ sum, const int* __restrict__ flag, int* __restrict__ out, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        out[i] = flag[i] == 1 ? isqrt_u16(sum[i]) : rms_div(sum[i], recip32((unsigned)flag[i]));
}

cudaError_t launch_rms(const int* sum, const int* flag, int* out, int n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int blocks = (n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096;
    rms_kernel<<<blocks, 256, 0, s>>>(sum, flag, out, n);
    return cudaGetLastError();
}

cudaError_t launch_tile_map(const ImgDesc* imgs, int nimg, int total_tiles, int* tile_img, cudaStream_t s) {
    if (nimg <= 0) return cudaSuccess;
    tile_map_kernel<<<(unsigned)nimg, 256, 0, s>>>(imgs, nimg, total_tiles, tile_img);
    return cudaGetLastError();
}

}  // namespace hg
