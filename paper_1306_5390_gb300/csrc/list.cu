// List passes: passes of Algorithms 1-2 that evaluate only the pixels that
// can differ from what their output canvas already holds, all run by one
// persistent (cooperative) launch.
//
// Write I_t for the image after pass t.  Pass t + 1 reads I_t (canvas `cur`)
// and turns canvas `aux`, which holds I_(t-1), into I_(t+1).  A pixel's value
// in I_(t+1) depends only on its (2 beta + 1)^2 window in I_t, exactly as its
// value in I_(t-1) depended on that window in I_(t-2).  So a pixel q must be
// evaluated only if its window holds a pixel where I_t differs from I_(t-2);
// everywhere else I_(t+1)(q) = I_(t-1)(q) is in place already.  The list a
// pass reads is therefore D_t = {p : I_t(p) != I_(t-2)(p)}: the owner of q
// compares its new value with the one it finds in `aux` and, if they differ,
// writes it and appends q to D_(t+1).  Pixels that alternate between two
// values (a large part of the impulses never settles in another way) leave
// the lists, and the lists shrink by a factor of two to three per pass instead
// of staying at the number of oscillating pixels (8192 x 8192, 30 %
// impulses, beta 1: 24 passes evaluate 1.1 M pixels instead of 13.4 M, 0.164 ms
// instead of 0.315; beta 2, 28 passes: 10.3 M instead of 21.4 M, 0.320 ms instead
// of 0.520; 1920 x 1080, beta 2: 0.078 ms instead of 0.180).
//
// The first pass reads the fused launch's list C_t = {p : I_t(p) != I_(t-1)(p)}.
// It serves as well (a pixel with no such p in its window keeps I_t(q) =
// I_(t-1)(q)), and a pass that reads C_t finds every pixel of C_(t+1) and of
// D_(t+1) and can make either; a pass that reads D_t can make only D_(t+1).  D_t
// holds C_(t-1)'s settled pixels too, so while the changes still die out C is the
// shorter list.  make_c draws the line: C again while the last list was
// shorter than 3/4 (short lists 3/5) of the one before it (beta 5, 1000 x
// 1500, 2 % impulses: 1.5 M evaluations against 2.8 M with D from the first
// pass on); the first pass, which knows no ratio, makes D when the fused
// launches ran kDirectD passes, by then the changes left are mostly
// oscillations.  (3/4 for lists of some thousand pixels too: 1024 x 1024, 70 %
// impulses, beta 2, 75 us against 70; 3/5 for all: textured 4096 x 4096, alpha 1,
// beta 3, 3.31 ms against 3.13.)  Lists of more than 1/32 of the pixels are no
// oscillations yet: they make C while they shrink at all (70 % impulses,
// textured 8192 x 8192, alpha 2, beta 1: 6.28 ms a call against 7.40 when D began at
// once; 4096 x 4096, alpha 2, beta 3: 1.69 against 2.15, 23 % slower with the line
// at 1/16; with 1/64 8192 x 8192, alpha 10 is 9 % slower), and with alpha 0, which
// replaces every interior pixel in every pass, however they shrink (1024 x
// 1024, beta 1: 0.65 ms against 0.75).
//
// k and the converged flag need to know whether a pass changed the image,
// N_t = #{q : I_t(q) != I_(t-1)(q)} > 0.  For a pixel that is not evaluated
// the inequality holds for pass t + 1 as it did for pass t, so N_(t+1) = N_t
// + sum over the evaluated q of [I_(t+1)(q) != I_t(q)] - [I_t(q) !=
// I_(t-1)(q)].  (A pass that reads C_t evaluates every changed pixel: the first
// terms alone.)  When a D list comes out empty, the image alternates
// between the two canvases for good: N = 0 means that the passes before this
// one and its predecessor were the last to change anything, N > 0 that every
// further pass changes the image, so k = max_k and the parity of the passes
// left names the canvas.
//
// Every pixel q within beta of a listed pixel is evaluated once, by the listed
// pixel p that "owns" q: the first one, in raster order, of q's window (read
// from the list's bitmap).  For beta 1 one thread takes one listed pixel
// p, loads its 5 x 5 neighbourhood and evaluates the pixels of p's 3 x 3 window
// that p owns from registers.  For wider windows one thread takes one (listed
// pixel, window row) pair, decides ownership for the whole row from one
// bitmap word per window row, and queues the owned pixels in shared memory;
// the CTA then evaluates its queue with all threads, so the evaluations run
// without idle lanes.  When a list overflowed its capacity, the pass evaluates
// every pixel instead.
//
// Passes are separated by a grid-wide barrier (all CTAs are co-resident, by
// cooperative launch).  Every CTA tracks k, the list lengths and the
// current canvas itself from values that are final at the barrier, so one
// barrier per pass suffices; four list/bitmap sets rotate so that each set
// is reset or cleared only while no CTA can still touch it.  Short lists are
// left to CTA 0 alone (solo_passes), which needs no grid barrier between its
// passes.  Waits at the
// barrier are bounded: after one to two seconds the kernel records an error and
// returns, and the call reports HGRMS_ETIMEOUT.
#include "common.cuh"
#include "kernels.h"

namespace hg {

namespace {

constexpr int kListThreads = 512;

// Loads of the bitmaps and canvases that the previous pass wrote go through
// L1 (__ldca): nearby evaluations of one CTA read overlapping windows, and an
// L2-only load moves a whole 32-byte sector per 4-byte word.  This is
// coherent because every pass starts after the grid barrier, whose
// gpu-scope acquire (thread 0) and CTA barrier order each thread's later
// loads after every write of the previous pass - the pattern of a grid-wide
// synchronisation, after which ordinary loads observe the other CTAs' writes.
// Nothing a pass reads through L1 is written during the same pass; the output
// canvas, which a pass reads and writes, is read from L2 (__ldcg).

// Bits [start, start + N) of a bitmap row in the low bits (outside [0, 32 *
// nwords): 0; bits from N on are not defined).  The second word is loaded only
// where the bits reach it.
template <int N>
__device__ __forceinline__ uint32_t row_bits(const uint32_t* __restrict__ row, int nwords, int start) {
    static_assert(N <= 32, "one word of bits");
    const int w0 = start >= 0 ? (start >> 5) : -((31 - start) >> 5);
    const int sh = start - 32 * w0;
    const uint32_t a = (w0 >= 0 && w0 < nwords) ? __ldca(row + w0) : 0u;
    const uint32_t b = (sh > 32 - N && w0 + 1 >= 0 && w0 + 1 < nwords) ? __ldca(row + w0 + 1) : 0u;
    return __funnelshift_r(a, b, (uint32_t)sh);
}

// Algorithm 2 for an interior pixel (card <= 2 is implied by flag >
// pix_count - 3 for alpha >= 1, and card is 0 for alpha = 0).  `p` points at
// the pixel in a row-major byte array with row stride `stride`.
template <int B>
__device__ __forceinline__ int eval_pixel(const uint8_t* p, long long stride, int alpha) {
    const int ip = p[0];
    int sum = 0, flag = 0;
#pragma unroll
    for (int dy = -B; dy <= B; ++dy)
#pragma unroll
        for (int dx = -B; dx <= B; ++dx) {
            const int v = p[dy * stride + dx];
            const bool open = !(v < ip + alpha + 1 && v > ip - alpha);
            sum += open ? v * v : 0;
            flag += open ? 1 : 0;
        }
    constexpr int kPixCount = (2 * B + 1) * (2 * B + 1);
    if (flag > kPixCount - 3) return rms_window<B>(sum, flag);
    return ip;
}

// Byte mask (0xFF per byte) of the bytes v_j of v with lo <= v_j <= hi, for
// kl = (256 - lo) and kh = (256 - (hi + 1)) in both 16-bit halves, 0 <= lo <=
// 256 and 0 <= hi + 1 <= 256.  The even and the odd bytes are taken apart
// into 16-bit lanes; in a lane, byte + 256 - lo lies in 0..511 and has bit 8
// set exactly when byte >= lo, and byte + 256 - (hi + 1) has it set exactly
// when byte > hi (no carry reaches the next lane).
__device__ __forceinline__ uint32_t bytes_in_range(uint32_t v, uint32_t kl, uint32_t kh) {
    const uint32_t e = v & 0x00FF00FFu, o = __byte_perm(v, 0u, 0x4341u);
    const uint32_t ce = (e + kl) & ~(e + kh);
    const uint32_t co = (o + kl) & ~(o + kh);
    return (((ce >> 8) & 0x00010001u) | (co & 0x01000100u)) * 0xFFu;
}

// Algorithm 2 for an interior pixel whose (2B + 1)^2 window is loaded as
// rows of bytes (win[r][j / 4] byte j % 4 = value at offset (r - B, j - B)),
// four values at a time: a value v is closed when ip - alpha < v <= ip +
// alpha (bytes_in_range with lo = max(ip - alpha + 1, 0), hi = min(ip +
// alpha, 255); for alpha = 0 nothing is); the open values' squares sum in
// one 4-way dot product per word and a second one with 0x01010101 counts
// the open values (255 each).  For beta 2 the fifth value of each
// row is gathered four rows to a word first.  Returns the new value (ip when
// the pixel is not replaced; card <= 2 is implied by flag > pix_count - 3
// for alpha >= 1, and card is 0 for alpha = 0).
template <int B>
__device__ __forceinline__ int eval_window(const uint32_t (&win)[2 * B + 1][(2 * B + 4) / 4], int alpha) {
    constexpr int W = 2 * B + 1, NW = (W + 3) / 4, P = W * W;
    const int ip = (int)((win[B][B / 4] >> (8 * (B % 4))) & 0xffu);
    const int lo = max(ip - alpha + 1, 0), hi = min(ip + alpha, 255);
    const uint32_t kl = 0x01000100u - (uint32_t)lo * 0x00010001u;
    const uint32_t kh = 0x01000100u - (uint32_t)(hi + 1) * 0x00010001u;
    unsigned sum = 0u, open255 = 0u;  // 255 per open value
    auto word = [&](uint32_t v, uint32_t ok) {
        const uint32_t open = ~bytes_in_range(v, kl, kh) & ok;
        sum = __dp4a(v & open, v, sum);
        open255 = __dp4a(open, 0x01010101u, open255);
    };
    if constexpr (B == 2) {
        // Values -2..1 of every row, then the values +2 of rows 0-3 in one word and of row 4.
#pragma unroll
        for (int r = 0; r < W; ++r) word(win[r][0], 0xFFFFFFFFu);
        const uint32_t t01 = __byte_perm(win[0][1], win[1][1], 0x0040u);
        const uint32_t t23 = __byte_perm(win[2][1], win[3][1], 0x0040u);
        word(__byte_perm(t01, t23, 0x5410u), 0xFFFFFFFFu);
        word(win[4][1], 0x000000FFu);
    } else {
#pragma unroll
        for (int r = 0; r < W; ++r)
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                constexpr int kLast = W - 4 * (NW - 1);  // values in the last word of a row
                const uint32_t ok = (k < NW - 1 || kLast == 4) ? 0xFFFFFFFFu : ((1u << (8 * kLast)) - 1u);
                word(win[r][k], ok);
            }
    }
    if (open255 <= 255u * (P - 3)) return ip;
    const unsigned m = open255 == 255u * P ? recip32(P) : (open255 == 255u * (P - 1) ? recip32(P - 1) : recip32(P - 2));
    return rms_div((int)sum, m);
}

// Grid-wide barrier over co-resident CTAs that also sums one count over all
// CTAs (*count: this CTA's contribution, in shared memory; *total receives
// the sum).  Barrier number b (1, 2, ...) uses counter (b & 1), a 64-bit
// word whose low half counts arrivals and whose high half accumulates the
// counts.  Each CTA arrives with one release reduction (no value returned,
// so no round trip) and polls its counter until the low half reaches the
// barrier's target; counters are never reset within a call, so the target
// of the n-th use of a counter is n * nblocks (plus `extra`, which only the
// test of the bounded wait sets: an arrival that never comes).  The high half's growth since
// this counter's previous use is this barrier's sum: a CTA can arrive at the
// next barrier of the same counter only after every CTA has passed the
// barrier in between, hence after every CTA has read this one's value.  The
// wait is bounded; returns false (for every thread of the CTA) when it gave
// up.
__device__ __forceinline__ bool grid_barrier(GridBar* b, Ctrl* c, unsigned nblocks, unsigned& nbar,
                                             const unsigned* count, unsigned (&prev_hi)[2], unsigned& total,
                                             unsigned extra, unsigned max_spins) {
    __shared__ unsigned s_total;
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0) {
        const unsigned bn = nbar + 1u;
        const unsigned par = bn & 1u;
        unsigned long long* ctr = &b->ctr[par].v;
        const unsigned long long add = 1ull + ((unsigned long long)*count << 32);
        const unsigned target = ((bn + 1u) >> 1) * nblocks + extra;  // uses of this counter so far x CTAs
        // No separate fence: the CTA barrier above orders every thread's
        // writes of this pass before thread 0's release reduction, and a
        // release is cumulative (it makes visible at gpu scope what its
        // thread has observed, here through the CTA barrier), so a CTA whose
        // acquire load sees this arrival sees those writes too.  (A fence
        // here measured 4-7 % of the list passes on 8192 x 8192.)
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(ctr), "l"(add) : "memory");
        unsigned spins = 0;
        unsigned long long v = 0;
        while (true) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(ctr) : "memory");
            if ((unsigned)v >= target) break;
            if (++spins > max_spins) {  // built-in limit 2^22: one to two seconds
                atomicExch(&c->error, 1u);
                ok = 0;
                break;
            }
            if (spins > 16) __nanosleep(64);
        }
        const unsigned hi = (unsigned)(v >> 32);
        s_total = ok ? hi - prev_hi[par] : 0u;
        prev_hi[par] = hi;
        nbar = bn;
    }
    ok = __syncthreads_and(ok);
    total = s_total;
    return ok != 0;
}

// W bytes of a canvas row starting at p, realigned into ((W + 3) / 4)
// words (byte j at bits 8 (j % 4) of word j / 4; bytes from W on are not
// defined); reads whole aligned words, which the canvas padding keeps in
// bounds, and no more of them than can hold the W bytes (for beta 2 two
// instead of three: the passes of long lists are bound by their loads).
template <int W>
__device__ __forceinline__ void load_row_bytes(const uint8_t* p, uint32_t (&r)[(W + 3) / 4]) {
    constexpr int NW = (W + 3) / 4, NL = (W + 3 + 3) / 4;
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    const uint32_t* q = reinterpret_cast<const uint32_t*>(a & ~uintptr_t(3));
    const uint32_t sh = (uint32_t)(a & 3u) * 8u;
    uint32_t w[NW + 1];
#pragma unroll
    for (int i = 0; i <= NW; ++i) w[i] = i < NL ? __ldca(q + i) : 0u;
#pragma unroll
    for (int i = 0; i < NW; ++i) r[i] = __funnelshift_r(w[i], w[i + 1], sh);
}

// Warp-collective: set the bit of `img` in the CTA's changed-image bitmap
// for every lane with `ch` (one shared atomic per distinct image).
__device__ __forceinline__ void mark_image(uint32_t* bits, bool ch, unsigned img, int lane) {
    const unsigned bal = __ballot_sync(0xffffffffu, ch);
    if (!bal) return;
    const unsigned peers = __match_any_sync(0xffffffffu, ch ? img : 0xffffffffu);
    if (ch && (int)(__ffs(peers & bal) - 1) == lane) atomicOr(bits + (img >> 5), 1u << (img & 31));
}

// The three bytes p[0..2] of the output canvas, from L2.
__device__ __forceinline__ uint32_t load3_cg(const uint8_t* p) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    const uint32_t* q = reinterpret_cast<const uint32_t*>(a & ~uintptr_t(3));
    return __funnelshift_r(__ldcg(q), (a & 3u) > 1u ? __ldcg(q + 1) : 0u, (uint32_t)(a & 3u) * 8u);
}

// Warp-collective: img_n[img] += d for every lane with d != 0 (one atomic per
// distinct image).
__device__ __forceinline__ void add_image(int* img_n, int d, unsigned img, int lane) {
    if (!__any_sync(0xffffffffu, d != 0)) return;
    const unsigned peers = __match_any_sync(0xffffffffu, d != 0 ? img : 0xffffffffu);
    const int sum = __reduce_add_sync(peers, d);
    if (d != 0 && sum != 0 && __ffs(peers) - 1 == lane) atomicAdd(img_n + img, sum);
}

// Short lists.  A pass of a handful of pixels is all latency.  Lists whose
// (listed pixel, window position) pairs fit the grid's threads take the direct
// path, one round of loads and one evaluation per thread (beta 1 and 2; for
// wider windows most of the pairs would load for nothing): 8192 x 8192, beta 1,
// 3.8-5 us a pass where a thread with nine positions in turn took 6.3-7.3, of
// which the barrier is about 2 us.  Lists of at most kSoloPixels pixels are
// left to CTA 0 alone, with the lists and the claims in shared memory: 1.25 us
// a pass for 30 pixels of beta 2, 2.4 us for 44, 5.4 us for 205 of beta 1 (four
// rounds of the CTA's threads, where the grid is faster again).  kSoloPixels: twice as many
// for beta 1 cost 8192 x 8192 20 us more a call, half as many 64 photographs 8 us and
// 1000 x 1000 3 us; for beta 2 and 3 (four rounds) half as many measured the
// same on 700 x 900 to 8192 x 8192.  kDescCache: 64 and 256 entries measured like
// 128 on batches of 64 to 512 images (128 take 6 KB).  kDirectD lies between
// beta 2's four fused passes (8192 x 8192 0.94 ms a call; 1.00 with D in the first
// list pass) and beta 1's eight, where D gains on one image and photographs
// (0.914 against 0.918 ms, 0.599 against 0.604) and loses on uneven ones (128 of
// them 3.00 ms against 2.95).
constexpr unsigned kDirectD = 6;
constexpr int kDirectB = 2;
constexpr int kDescCache = 128;
constexpr int kSoloEvals = 2048;
template <int B>
constexpr unsigned kSoloPixels = B == 1 ? 112u : (unsigned)(kSoloEvals / ((2 * B + 1) * (2 * B + 1)));
constexpr int kSoloHash = 2 * kSoloEvals;        // claim table, at most half full
constexpr int kSoloPasses = 1024;                // then the other CTAs' waits end
constexpr unsigned kSoloClear = 1u << 16;        // largest list whose bitmap CTA 0 clears

}  // namespace

// State of the passes that every CTA follows (see the header).
struct LoopState {
    int t;              // passes run by the whole grid (set rotation)
    unsigned k;         // number of the last pass run
    unsigned cur, aux;  // canvases of I_t and I_(t-1)
    unsigned n_cur;     // entries of the list the next pass reads
    unsigned n_last;    // entries of the list before it (its bitmap is cleared by the next pass)
    unsigned n_before;  // entries of the list that the last pass read (0: no pass yet)
    bool c_list;        // the next pass reads C_t (else D_t)
    // Whether the next pass, from a list of n entries, makes C (see the header;
    // k0: passes before this launch, dense: 1/32 of the pixels).
    __device__ __forceinline__ bool make_c(unsigned n, unsigned k0, unsigned dense, int alpha) const {
        if (!c_list) return false;
        const unsigned long long now = n, before = n_before;
        if (n > dense && (n_before == 0u || now * 16u < before * 15u || (alpha == 0 && n / 4u > dense))) return true;
        return n_before == 0u ? k0 < kDirectD : (n > kShortList ? now * 4u < before * 3u : now * 5u < before * 3u);
    }
};

// Passes run by CTA 0 alone, from a list of st.n_cur <= kSoloPixels<B>
// pixels, until a list comes out empty, k reaches max_k, a list is longer
// than that or kSoloPasses passes have run (the other CTAs wait meanwhile, and
// their wait is bounded).  One thread takes one (listed pixel, window
// position) pair and claims its pixel in a hash table.  Lists and claims
// live in shared memory; the change sets are left as the grid's passes
// expect them: the list of the next pass in the set that held the first one,
// every other bitmap empty (st.t and the append counters stand still; another
// CTA may not have read them yet).  st is updated (thread-uniform); s_n is two
// counters; dn accumulates this thread's share of the change of N.
template <int B, bool kBatch>
__device__ __forceinline__ void solo_passes(const PassArgs& a, const ImgDesc& one, const int base, const int xb,
                                            const int yb, const unsigned max_k, const unsigned k0, LoopState& st, uint32_t* lists,
                                            uint32_t* hash, unsigned* s_n, unsigned& evals, int& dn) {
    constexpr int W = 2 * B + 1, P = W * W, NW = (W + 3) / 4;
    static_assert(kSoloPixels<B> * P <= kSoloEvals, "the next list and the claim table hold every window position");
    const int tid = threadIdx.x;
    uint32_t* list = lists;
    uint32_t* next = lists + kSoloEvals;
    {
        // The list, and clean bitmaps for all sets.
        const int si = (st.t + base) & 3, sc = (st.t + base + 3) & 3;
        auto clear = [&](uint32_t* bm, uint32_t e) {
            unsigned img;
            int y, x;
            unpack_entry(e, xb, yb, img, y, x);
            const ImgDesc d = kBatch ? load_desc(a.imgs, img) : one;
            bm[d.bm_off + (long long)y * d.bm_words + (x >> 5)] = 0u;
        };
        for (unsigned i = tid; i < st.n_cur; i += kListThreads) {
            const uint32_t e = __ldcg(a.lists[si] + i);
            list[i] = e;
            clear(a.bitmaps[si], e);
        }
        for (unsigned i = tid; i < st.n_last; i += kListThreads) clear(a.bitmaps[sc], __ldcg(a.lists[sc] + i));
    }
    unsigned n = st.n_cur;
    for (int passes = 1;; ++passes) {
        for (int i = tid; i < kSoloHash; i += kListThreads) hash[i] = 0xffffffffu;
        unsigned* nn = s_n + (passes & 1);  // the other one may still be read
        if (tid == 0) *nn = 0u;
        __syncthreads();
        const uint8_t* in_arena = a.canvas[st.cur];
        uint8_t* out_arena = a.canvas[st.aux];
        const int ntask = (int)n * P;
        const bool make_c = st.make_c(n, k0, a.list_dense, a.alpha);
        for (int i = tid; i < ntask; i += kListThreads) {
            const int e = i / P, o = i - e * P;
            unsigned img;
            int y, x;
            unpack_entry(list[e], xb, yb, img, y, x);
            const ImgDesc d = kBatch ? load_desc(a.imgs, img) : one;
            y += o / W - B;
            x += o % W - B;
            if (y < B || y >= d.rows - B || x < B || x >= d.cols - B) continue;
            // Claim q (an interior pixel never packs to the empty key: its row
            // and column are not the last ones of the fields' ranges).
            const uint32_t key = pack_entry(img, y, x, xb, yb);
            unsigned slot = (key * 0x9E3779B1u) >> 16 & (kSoloHash - 1);
            bool mine = false;
            for (int probe = 0; probe < kSoloHash; ++probe) {
                const uint32_t was = atomicCAS(&hash[slot], 0xffffffffu, key);
                mine = was == 0xffffffffu;
                if (mine || was == key) break;
                slot = (slot + 1) & (kSoloHash - 1);
            }
            if (!mine) continue;
            const long long off = d.off + (long long)(kPadY + y) * d.pitch + kPadX + x;
            const uint8_t* in = in_arena + off;
            const int was = __ldcg(out_arena + off);
            uint32_t win[W][NW];
#pragma unroll
            for (int r = 0; r < W; ++r) load_row_bytes<W>(in + (long long)(r - B) * d.pitch - B, win[r]);
            ++evals;
            const int ip = (int)((win[B][B / 4] >> (8 * (B % 4))) & 0xffu);
            const int nv = eval_window<B>(win, a.alpha);
            if (nv != was) out_arena[off] = (uint8_t)nv;
            if (nv != (make_c ? ip : was)) next[atomicAdd(nn, 1u)] = key;
            const int now = nv != ip ? 1 : 0, before = ip != was ? 1 : 0;
            const int delta = (make_c ? 0 : now) - (st.c_list ? 0 : before);
            dn += delta;
            if (kBatch && a.img_k) {
                if (delta) atomicAdd(a.img_n + img, delta);
                if (now || before) atomicMax(a.img_k + img, st.k + (unsigned)now);
            }
        }
        __syncthreads();
        st.n_before = n;
        n = *nn;
        ++st.k;
        st.c_list = make_c;
        const unsigned c = st.cur;
        st.cur = st.aux;
        st.aux = c;
        uint32_t* l = list;
        list = next;
        next = l;
        if (n == 0u || st.k >= max_k || n > kSoloPixels<B> || passes >= kSoloPasses) break;
    }
    st.n_cur = n;
    st.n_last = 0u;
    if (n != 0u && st.k < max_k) {
        // The grid goes on from this list.
        const int si = (st.t + base) & 3;
        for (unsigned i = tid; i < n; i += kListThreads) {
            const uint32_t e = list[i];
            if (i < a.list_cap) a.lists[si][i] = e;
            unsigned img;
            int y, x;
            unpack_entry(e, xb, yb, img, y, x);
            const ImgDesc d = kBatch ? load_desc(a.imgs, img) : one;
            atomicOr(a.bitmaps[si] + d.bm_off + (long long)y * d.bm_words + (x >> 5), 1u << (x & 31));
        }
    }
}

// kBatch = false: one image, described by the launch arguments (pitch, rows,
// cols, bm_words; entries packed 16/16); true: the image table.
template <int B, bool kBatch>
__global__ void __launch_bounds__(kListThreads, 2) list_loop_kernel(PassArgs a) {
    constexpr int W = 2 * B + 1, P = W * W;
    constexpr int kWarps = kListThreads / 32;
    __shared__ int s_np;
    __shared__ unsigned s_k, s_cur, s_aux, s_maxk, s_base;
    __shared__ unsigned s_n, s_nclr, s_app, s_solo_n[2];
    __shared__ int s_dn;
    // Staged list entries, one buffer per warp; solo passes keep their two lists here.
    __shared__ uint32_t stage_all[kWarps * StagedList::kCap];
    static_assert(kWarps * StagedList::kCap >= 2 * kSoloEvals, "the solo lists fit the staging buffers");
    __shared__ int s_counts[kWarps + 1];
    __shared__ unsigned long long s_evals;
    // Images changed by this pass, and by the pass before it (both as this CTA saw).
    __shared__ uint32_t s_imgbits[kBatch ? kMaxBatchImages / 32 : 1], s_imgbits0[kBatch ? kMaxBatchImages / 32 : 1];
    // Pixels this CTA evaluates in the current chunk (beta >= 2); the claim table of the solo passes.
    constexpr int kQueue = B == 1 ? 1 : kListThreads * W;
    __shared__ uint32_t s_queue[kQueue > kSoloHash ? kQueue : kSoloHash];
    __shared__ int s_qn[2];  // queue lengths; chunks alternate between them
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    Ctrl* ctrl = a.ctrl;
    if (tid == 0) {
        s_evals = 0ull;
        s_qn[0] = 0;
        s_qn[1] = 0;
        s_np = launch_passes(ctrl, 1);
        s_k = __ldcg(&ctrl->k);
        s_cur = __ldcg(&ctrl->cur);
        s_aux = __ldcg(&ctrl->aux);
        s_maxk = __ldcg(&ctrl->max_k);
        // The last fused launch wrote change set (fused launches - 1) % 4.
        s_base = (__ldcg(&ctrl->fused_work) + 3u) & 3u;
    }
    if constexpr (kBatch)
        for (int i = tid; i < kMaxBatchImages / 32; i += kListThreads) s_imgbits[i] = s_imgbits0[i] = 0u;
    __syncthreads();
    if (s_np == 0) return;  // the fused launch already finished the call
    LoopState st;
    st.t = 0;
    st.k = s_k;
    st.cur = s_cur;
    st.aux = s_aux;
    st.c_list = true;
    st.n_before = 0u;
    unsigned gen = 0u;               // thread 0: barriers completed; the barrier struct is zeroed at the start of every call
    unsigned prev_hi[2] = {0u, 0u};  // thread 0: counts seen at the last use of each barrier counter
    const int base = (int)s_base;
    const unsigned max_k = s_maxk, k0 = s_k;
    const unsigned max_spins = a.bar_spins ? a.bar_spins : (1u << 22);
    bool failed = false;
    unsigned evals = 0;
    int qpar = 0;  // queue counter of the next chunk (CTA-uniform)
    const long long gthreads = (long long)gridDim.x * blockDim.x;
    const long long gtid = (long long)blockIdx.x * blockDim.x + tid;
    const long long warp_base = (long long)blockIdx.x * blockDim.x + (tid & ~31);
    // Tasks are dealt to the CTAs a warp at a time: neighbours on a list are
    // mostly neighbours in the image, and a warp's loads then share cache
    // lines (a load of 32 lanes in 32 lines takes 32 turns in L1).  64
    // photographs, first pass of 195,000 listed pixels: 25 us, 40 us when every
    // lane went to another CTA.
    const long long first_task = ((long long)warp * gridDim.x + blockIdx.x) * 32 + lane;
    // The single image as a table entry (its offsets are 0).
    ImgDesc one;
    if constexpr (!kBatch) {
        one.off = 0;
        one.bm_off = 0;
        one.pitch = (int)a.pitch;
        one.rows = a.rows;
        one.cols = a.cols;
        one.tiles_x = 0;
        one.tile0 = 0;
        one.bm_words = a.bm_words;
        one.user = nullptr;
    }
    // Batches: the first images' table entries in shared memory (every barrier
    // empties L1, so a table read costs a pass one more trip to L2).
    constexpr int kCached = kBatch && B <= 4 ? kDescCache : 0;
    __shared__ ImgDesc s_desc[kCached > 0 ? kCached : 1];
    if constexpr (kCached > 0) {
        for (int i = tid; i < min(a.nimg, kCached); i += kListThreads) s_desc[i] = load_desc(a.imgs, (unsigned)i);
    }
    auto desc = [&](unsigned img) -> ImgDesc {
        if constexpr (!kBatch) return one;
        else return img < (unsigned)kCached ? s_desc[img] : load_desc(a.imgs, img);
    };
    constexpr int kXb = 16, kYb = 16;
    const int xb = kBatch ? a.xb : kXb, yb = kBatch ? a.yb : kYb;
    StagedList sl{stage_all + warp * StagedList::kCap, 0, 0u};
    // List lengths at the start; later ones come from the barrier.
    if (tid == 0) {
        s_n = __ldcg(&ctrl->list_n[base]);
        s_nclr = __ldcg(&ctrl->list_n[(base + 3) & 3]);
        s_app = 0u;
        s_dn = 0;
    }
    __syncthreads();
    st.n_cur = s_n;
    st.n_last = s_nclr;

    while (true) {
        int dn = 0;  // this thread's share of the change of N
        if (st.n_cur <= kSoloPixels<B> && st.n_cur <= a.list_cap && st.n_last <= kSoloClear &&
            st.n_last <= a.list_cap) {
            if (blockIdx.x == 0) {
                solo_passes<B, kBatch>(a, one, base, xb, yb, max_k, k0, st, stage_all, s_queue, s_solo_n, evals, dn);
                dn = __reduce_add_sync(0xffffffffu, dn);
                if (lane == 0 && dn) atomicAdd(&s_dn, dn);
                __syncthreads();
                if (tid == 0) {
                    s_qn[0] = s_qn[1] = 0;
                    if (s_dn) atomicAdd(&ctrl->n_diff, s_dn);
                    s_dn = 0;
                    // The entry of the barrier ahead, by its parity: it is
                    // written again two barriers on at the earliest, and every
                    // CTA reaches the one in between after its reads below.
                    auto& e = ctrl->solo[gen & 1u];
                    e.k = st.k;
                    e.n = st.n_cur;
                    e.before = st.c_list ? st.n_before : 0xffffffffu;
                }
            }
            unsigned zero = 0;
            if (!grid_barrier(a.bar, ctrl, gridDim.x, gen, &s_app, prev_hi, zero, a.bar_extra, max_spins)) {
                failed = true;
                break;
            }
            if (blockIdx.x != 0) {
                if (tid == 0) {
                    const auto& e = ctrl->solo[(gen & 1u) ^ 1u];  // the barrier counted itself
                    s_k = __ldcg(&e.k);
                    s_n = __ldcg(&e.n);
                    s_nclr = __ldcg(&e.before);
                }
                __syncthreads();
                const unsigned ran = s_k - st.k;
                st.k = s_k;
                st.n_cur = s_n;
                st.n_last = 0u;
                st.n_before = s_nclr;
                st.c_list = s_nclr != 0xffffffffu;
                if (ran & 1u) {
                    const unsigned c = st.cur;
                    st.cur = st.aux;
                    st.aux = c;
                }
            }
            if (st.n_cur == 0u || st.k >= max_k) break;
            continue;
        }
        const int si = (st.t + base) & 3, so = (st.t + base + 1) & 3, sc = (st.t + base + 3) & 3;
        const uint8_t* in_arena = a.canvas[st.cur];
        uint8_t* out_arena = a.canvas[st.aux];
        const uint32_t* prev = a.lists[si];
        const uint32_t* bm_prev = a.bitmaps[si];
        uint32_t* next = a.lists[so];
        uint32_t* bm_next = a.bitmaps[so];
        unsigned* nnext = &ctrl->list_n[so];
        const bool make_c = st.make_c(st.n_cur, k0, a.list_dense, a.alpha);
        // N is needed from the first D_t on: the pass that makes it counts the
        // pixels it changes, the later ones the differences.
        const int add = make_c ? 0 : 1, sub = st.c_list ? 0 : 1;
        if (tid == 0 && blockIdx.x == 0) {
            // Set (t + base + 2) % 4 is next written by pass t + 1; its list
            // was last read (to clear its bitmap) in pass t - 1.
            ctrl->list_n[(st.t + base + 2) & 3] = 0u;
        }
        const unsigned n = st.n_cur, nclr = st.n_last;
        // The windows of a sixteenth of the pixels hold most of them: for beta
        // >= 2 a pass over every pixel costs less than one by such a list.  Lines at
        // 1/8, 1/16 and 1/32 of the pixels: textured 4096 x 4096, alpha 1, beta 3,
        // 30 % impulses 3.03, 2.39 and 2.41 ms a call, alpha 2, beta 2, 70 % 1.38, 1.18
        // and 1.24; for beta 1 1/8 measured like the overflow alone.
        const bool whole = n > a.list_cap || (B > 1 && n / 2u > a.list_dense);
        // A short list: one thread per (listed pixel, window position).
        const bool direct = B <= kDirectB && (long long)n * P <= gthreads && !whole;
        // The list entry of this thread's first task, loaded before the bitmap clearing below so that the two
        // loads overlap.
        uint32_t pk_first = 0u;
        if (!whole) {
            const long long i0 = first_task;
            const long long per = direct ? P : (B == 1 ? 1 : W);
            if (i0 < (long long)n * per) pk_first = __ldcg(prev + (unsigned)(i0 / per));
        }
        // Clear bitmap sc (written by pass t - 2, read by pass t - 1) for pass
        // t + 2: walk its list, or clear it all if the list overflowed or is
        // longer than the bitmap.
        {
            const uint32_t* clr = a.lists[sc];
            uint32_t* bm_clr = a.bitmaps[sc];
            if (nclr <= a.list_cap && nclr <= a.bm_total) {
                for (long long i = gtid; i < nclr; i += gthreads) {
                    unsigned img;
                    int y, x;
                    unpack_entry(clr[i], xb, yb, img, y, x);
                    const ImgDesc d = desc(img);
                    bm_clr[d.bm_off + (long long)y * d.bm_words + (x >> 5)] = 0u;
                }
            } else {
                for (long long i = gtid; i < a.bm_total; i += gthreads) bm_clr[i] = 0u;
            }
        }
        if (B <= kDirectB && direct) {
            // Task (listed pixel p, window position): decides ownership of q
            // from the list's bits of q's window rows up to p's (as below),
            // and evaluates it, all from one round of loads.
            const unsigned i = (unsigned)first_task;
            bool ch = false, now = false, before = false;
            uint32_t v = 0;
            unsigned img = 0;
            if (i < n * (unsigned)P) {
                const int o = (int)(i % (unsigned)P);
                int py, px;
                unpack_entry(pk_first, xb, yb, img, py, px);
                const ImgDesc d = desc(img);
                const int dy = o / W - B, qy = py + dy, qx = px + o % W - B;
                if (qy >= B && qy < d.rows - B && qx >= B && qx < d.cols - B) {
                    const uint32_t* bmp = bm_prev + d.bm_off;
                    const uint8_t* in = in_arena + d.off + (long long)kPadY * d.pitch + kPadX;
                    const long long off = (long long)qy * d.pitch + qx;
                    uint8_t* out = out_arena + d.off + (long long)kPadY * d.pitch + kPadX + off;
                    constexpr int NW = (W + 3) / 4;
                    uint32_t win[W][NW];
                    const int was = __ldcg(out);
                    uint32_t ahead = 0u;  // listed pixels of q's window before p (bit j: column qx - B + j)
#pragma unroll
                    for (int r = 0; r < W; ++r) {
                        load_row_bytes<W>(in + off + (long long)(r - B) * d.pitch - B, win[r]);
                        const int gy = qy - B + r;
                        if (gy <= py) {
                            const uint32_t bits = row_bits<W>(bmp + (size_t)gy * d.bm_words, d.bm_words, qx - B) & ((1u << W) - 1u);
                            ahead |= gy < py ? bits : bits & ((1u << (px - qx + B)) - 1u);
                        }
                    }
                    if (ahead == 0u) {
                        ++evals;
                        const int ip = (int)((win[B][B / 4] >> (8 * (B % 4))) & 0xffu);
                        const int nv = eval_window<B>(win, a.alpha);
                        v = pack_entry(img, qy, qx, xb, yb);
                        if (nv != was) *out = (uint8_t)nv;
                        if (nv != (make_c ? ip : was)) {
                            ch = true;
                            atomicOr(bm_next + d.bm_off + (size_t)qy * d.bm_words + (qx >> 5), 1u << (qx & 31));
                        }
                        now = nv != ip;
                        before = ip != was;
                    }
                }
            }
            const int delta = (now ? add : 0) - (before ? sub : 0);
            dn += delta;
            if (kBatch && a.img_k) {
                mark_image(s_imgbits, now, img, lane);
                mark_image(s_imgbits0, before && !now, img, lane);
                add_image(a.img_n, delta, img, lane);
            }
            staged_append(sl, next, nnext, a.list_cap, ch, v, lane);
        } else if (!whole && B == 1) {
            // beta 1: one thread per listed pixel p.  It loads p's 5 x 5
            // neighbourhood, the 3 x 3 window of the output canvas and the
            // list's bits of the rows up to p's, and evaluates every pixel q
            // of p's 3 x 3 window that p owns (no listed pixel of q's window
            // precedes p in raster order) from those registers.
            long long i = first_task;
            uint32_t pk = pk_first;
            for (long long c0 = 0; c0 + 32ll * blockIdx.x < (long long)n; c0 += gthreads, i += gthreads) {
                const long long inext = i + gthreads;
                const uint32_t pk_next = inext < (long long)n ? __ldcg(prev + (unsigned)inext) : 0u;
                uint32_t chm = 0u;  // bit (dy + 1) * 3 + dx + 1: q = p + (dy, dx) goes on the next list
                int delta = 0;      // the change of N
                bool now = false, before = false;
                unsigned img = 0;
                int py = 0, px = 0;
                if (i < (long long)n) {
                    unpack_entry(pk, xb, yb, img, py, px);
                    const ImgDesc d = desc(img);
                    const uint32_t* bmp = bm_prev + d.bm_off;
                    const uint8_t* in = in_arena + d.off + (long long)kPadY * d.pitch + kPadX;
                    uint8_t* out = out_arena + d.off + (long long)kPadY * d.pitch + kPadX;
                    // List bits of rows py - 2 .. py, columns px - 2 .. (bit j: column px - 2 + j).
                    uint32_t rb[3];
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        const int gy = py - 2 + r;
                        rb[r] = gy >= 0 ? row_bits<5>(bmp + (size_t)gy * d.bm_words, d.bm_words, px - 2) : 0u;
                    }
                    // Rows py - 2 .. py + 2, bytes px - 2 .. px + 2 (the canvas padding keeps them in bounds).
                    uint32_t nb[5][2], ob[3];
                    const long long off = (long long)py * d.pitch + px;
#pragma unroll
                    for (int r = 0; r < 5; ++r) load_row_bytes<5>(in + off + (long long)(r - 2) * d.pitch - 2, nb[r]);
#pragma unroll
                    for (int r = 0; r < 3; ++r) ob[r] = load3_cg(out + off + (long long)(r - 1) * d.pitch - 1);
#pragma unroll
                    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
                        for (int dx = -1; dx <= 1; ++dx) {
                            const int qy = py + dy, qx = px + dx;
                            if (qy < 1 || qy >= d.rows - 1 || qx < 1 || qx >= d.cols - 1) continue;
                            // Ownership: q's window rows above p's hold no listed pixel,
                            // and p's row none left of p (bits dx + 1 .. 1).
                            bool owner = true;
#pragma unroll
                            for (int r = dy + 1; r <= dy + 3; ++r) {
                                if (r < 2 && (rb[r] & (7u << (dx + 1)))) owner = false;
                                if (r == 2 && (rb[2] & 3u & ~((1u << (dx + 1)) - 1u))) owner = false;
                            }
                            if (!owner) continue;
                            uint32_t w3[3][1];
#pragma unroll
                            for (int r = 0; r < 3; ++r)
                                w3[r][0] = __funnelshift_r(nb[dy + 1 + r][0], nb[dy + 1 + r][1], 8 * (dx + 1));
                            const int ip = (int)((w3[1][0] >> 8) & 0xffu);
                            const int was = (int)((ob[dy + 1] >> (8 * (dx + 1))) & 0xffu);
                            const int nv = eval_window<1>(w3, a.alpha);
                            ++evals;
                            if (nv != was) out[(long long)qy * d.pitch + qx] = (uint8_t)nv;
                            if (nv != (make_c ? ip : was)) {
                                chm |= 1u << ((dy + 1) * 3 + dx + 1);
                                atomicOr(bm_next + d.bm_off + (size_t)qy * d.bm_words + (qx >> 5), 1u << (qx & 31));
                            }
                            delta += (nv != ip ? add : 0) - (ip != was ? sub : 0);
                            if (kBatch) {
                                now = now || nv != ip;
                                before = before || ip != was;
                            }
                        }
                }
                dn += delta;
                if (kBatch && a.img_k) {
                    mark_image(s_imgbits, now, img, lane);
                    mark_image(s_imgbits0, before && !now, img, lane);
                    add_image(a.img_n, delta, img, lane);
                }
                // Append the pixels (one warp scan per round).
                staged_append_mask(sl, next, nnext, a.list_cap, chm, lane, [&](int bt) {
                    return pack_entry(img, py + bt / 3 - 1, px + bt % 3 - 1, xb, yb);
                });
                pk = pk_next;
            }
        } else if (!whole) {
            // Chunks of one task per thread: task (listed pixel p, window
            // row dy) finds the pixels q = p + (dy, dx) that p owns and
            // queues them in shared memory (phase A); the CTA then evaluates
            // its queue with every thread (phase B).
            const long long ntask = (long long)n * W;
            long long i = first_task;
            uint32_t pk = pk_first;  // later chunks' entries are loaded one chunk early
            for (long long c0 = 0; c0 + 32ll * blockIdx.x < ntask; c0 += gthreads, i += gthreads) {
                const long long inext = i + gthreads;
                const uint32_t pk_next = inext < ntask ? __ldcg(prev + (unsigned)(inext / W)) : 0u;
                // Phase A.  Ownership: no listed pixel of q's window precedes
                // p in raster order.  rb[r] = the list's bits in
                // row qy - B + r, columns px - 2B .. px + 2B (bit j: column
                // px - 2B + j); q = (qy, px + dx) has window columns bits
                // dx + B .. dx + 3B, its rows above py must have none and row
                // py none left of p (bits below 2B).
                unsigned own = 0u;  // bit dx + B: this task evaluates q
                unsigned img = 0;
                int py = 0, px = 0, qy = 0;
                if (i < ntask) {
                    const int dy = (int)(i % W) - B;
                    unpack_entry(pk, xb, yb, img, py, px);
                    const ImgDesc d = desc(img);
                    qy = py + dy;
                    if (qy >= B && qy < d.rows - B) {
                        const uint32_t* bmp = bm_prev + d.bm_off;
                        uint32_t rb[2 * B + 1];
#pragma unroll
                        for (int r = 0; r <= 2 * B; ++r) {
                            const int gy = qy - B + r;
                            rb[r] = (gy <= py) ? row_bits<4 * B + 1>(bmp + (size_t)gy * d.bm_words, d.bm_words, px - 2 * B) : 0u;
                        }
                        uint32_t ahead = 0u;
#pragma unroll
                        for (int r = 0; r <= 2 * B; ++r) {
                            const int gy = qy - B + r;
                            if (gy < py) ahead |= rb[r];
                            if (gy == py) ahead |= rb[r] & ((1u << (2 * B)) - 1u);
                        }
#pragma unroll
                        for (int dx = -B; dx <= B; ++dx) {
                            const int qx = px + dx;
                            const uint32_t wm = ((1u << W) - 1u) << (dx + B);
                            if (qx >= B && qx < d.cols - B && (ahead & wm) == 0u) own |= 1u << (dx + B);
                        }
                    }
                }
                {
                    // Queue the owned pixels (one shared atomic per warp).
                    const int cnt = __popc(own);
                    int incl = cnt;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int v = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += v;
                    }
                    const int wtot = __shfl_sync(0xffffffffu, incl, 31);
                    int wbase = 0;
                    if (lane == 31 && wtot) wbase = atomicAdd(&s_qn[qpar], wtot);
                    int pos = __shfl_sync(0xffffffffu, wbase, 31) + incl - cnt;
                    while (own) {
                        const int b = __ffs(own) - 1;
                        own &= own - 1u;
                        s_queue[pos++] = pack_entry(img, qy, px + b - B, xb, yb);
                    }
                }
                __syncthreads();
                // Phase B: Algorithm 2 for every queued pixel.
                const int qn = s_qn[qpar];
                // The other counter was last read before the previous chunk's
                // final barrier and is next used after this chunk's.
                if (tid == 0) s_qn[qpar ^ 1] = 0;
                for (int j0 = warp * 32; j0 < qn; j0 += kListThreads) {
                    const int j = j0 + lane;
                    bool ch = false, now = false, before = false;
                    uint32_t v = 0;
                    unsigned qimg = 0;
                    if (j < qn) {
                        int y, x;
                        v = s_queue[j];
                        unpack_entry(v, xb, yb, qimg, y, x);
                        const ImgDesc d = desc(qimg);
                        const uint8_t* in = in_arena + d.off + (long long)kPadY * d.pitch + kPadX;
                        constexpr int NW = (W + 3) / 4;
                        uint32_t win[W][NW];
                        const long long off = (long long)y * d.pitch + x;
                        uint8_t* out = out_arena + d.off + (long long)kPadY * d.pitch + kPadX + off;
                        const int was = __ldcg(out);
#pragma unroll
                        for (int r = 0; r < W; ++r) load_row_bytes<W>(in + off + (long long)(r - B) * d.pitch - B, win[r]);
                        ++evals;
                        const int ip = (int)((win[B][B / 4] >> (8 * (B % 4))) & 0xffu);
                        const int nv = eval_window<B>(win, a.alpha);
                        if (nv != was) *out = (uint8_t)nv;
                        if (nv != (make_c ? ip : was)) {
                            ch = true;
                            atomicOr(bm_next + d.bm_off + (size_t)y * d.bm_words + (x >> 5), 1u << (x & 31));
                        }
                        now = nv != ip;
                        before = ip != was;
                    }
                    const int delta = (now ? add : 0) - (before ? sub : 0);
                    dn += delta;
                    if (kBatch && a.img_k) {
                        mark_image(s_imgbits, now, qimg, lane);
                        mark_image(s_imgbits0, before && !now, qimg, lane);
                        add_image(a.img_n, delta, qimg, lane);
                    }
                    staged_append(sl, next, nnext, a.list_cap, ch, v, lane);
                }
                __syncthreads();  // every thread has read the queue
                qpar ^= 1;
                pk = pk_next;
            }
        } else {
            // Evaluate every pixel of every image.
            for (int im = 0; im < (kBatch ? a.nimg : 1); ++im) {
                const ImgDesc d = kBatch ? load_desc(a.imgs, (unsigned)im) : one;
                const uint8_t* in = in_arena + d.off + (long long)kPadY * d.pitch + kPadX;
                uint8_t* out = out_arena + d.off + (long long)kPadY * d.pitch + kPadX;
                const long long total = (long long)d.rows * d.cols;
                for (long long p0 = warp_base; p0 < total; p0 += gthreads) {
                    const long long i = p0 + lane;
                    bool ch = false, now = false, before = false;
                    uint32_t v = 0;
                    if (i < total) {
                        const int y = (int)(i / d.cols), x = (int)(i - (long long)y * d.cols);
                        const long long off = (long long)y * d.pitch + x;
                        ++evals;
                        const int ip = in[off], was = __ldcg(out + off);
                        int nv = ip;
                        if (y >= B && y < d.rows - B && x >= B && x < d.cols - B)
                            nv = eval_pixel<B>(in + off, d.pitch, a.alpha);
                        if (nv != was) out[off] = (uint8_t)nv;
                        if (nv != (make_c ? ip : was)) {
                            ch = true;
                            v = pack_entry((unsigned)im, y, x, xb, yb);
                            atomicOr(bm_next + d.bm_off + (size_t)y * d.bm_words + (x >> 5), 1u << (x & 31));
                        }
                        now = nv != ip;
                        before = ip != was;
                    }
                    const int delta = (now ? add : 0) - (before ? sub : 0);
                    dn += delta;
                    if (kBatch && a.img_k) {
                        mark_image(s_imgbits, now, (unsigned)im, lane);
                        mark_image(s_imgbits0, before && !now, (unsigned)im, lane);
                        add_image(a.img_n, delta, (unsigned)im, lane);
                    }
                    staged_append(sl, next, nnext, a.list_cap, ch, v, lane);
                }
            }
        }
        dn = __reduce_add_sync(0xffffffffu, dn);
        if (lane == 0 && dn) atomicAdd(&s_dn, dn);
        staged_flush(sl, next, nnext, a.list_cap, s_counts, kWarps);
        // Images this CTA saw changed by this pass (number k + 1) or the one
        // before it (staged_flush ends with a block barrier, so every mark is
        // in place).
        if (kBatch && a.img_k) {
            for (int w = tid; w < (a.nimg + 31) / 32; w += kListThreads) {
                const uint32_t now = s_imgbits[w];
                uint32_t bits = now | s_imgbits0[w];
                s_imgbits[w] = s_imgbits0[w] = 0u;
                while (bits) {
                    const int b = __ffs(bits) - 1;
                    bits &= bits - 1u;
                    atomicMax(a.img_k + 32 * w + b, st.k + ((now >> b) & 1u));
                }
            }
        }
        // Entries this CTA appended, and its share of the change of N.
        if (lane == 0 && sl.total) atomicAdd(&s_app, sl.total);
        sl.total = 0u;
        if (tid == 0) {
            if (s_dn) atomicAdd(&ctrl->n_diff, s_dn);  // s_dn is complete: staged_flush has block barriers
            s_dn = 0;
        }
        unsigned appended = 0;
        if (!grid_barrier(a.bar, ctrl, gridDim.x, gen, &s_app, prev_hi, appended, a.bar_extra, max_spins)) {
            failed = true;
            break;
        }
        if (tid == 0) s_app = 0u;  // read by thread 0 inside the barrier only
        ++st.t;
        ++st.k;
        st.c_list = make_c;
        st.n_before = st.n_cur;
        const unsigned c = st.cur;
        st.cur = st.aux;
        st.aux = c;
        st.n_last = st.n_cur;
        st.n_cur = appended;
        if (appended == 0u || st.k >= max_k) break;
    }
    const unsigned ev = __reduce_add_sync(0xffffffffu, evals);
    if (lane == 0 && ev) atomicAdd(&s_evals, (unsigned long long)ev);
    __syncthreads();
    if (tid == 0 && s_evals) atomicAdd(&ctrl->evals_list, s_evals);
    if (blockIdx.x != 0 || failed) return;
    // Every CTA holds the same state; the barriers order these writes after
    // every CTA's reads of the control block.
    // Whether the last pass changed the image.
    const bool still = st.c_list ? st.n_cur != 0u : __ldcg(&ctrl->n_diff) != 0;
    unsigned k = st.k;
    if (still && st.n_cur == 0u) {
        // The image alternates between the two canvases.
        if ((max_k - k) & 1u) st.cur = st.aux;
        k = max_k;
    } else if (!still) {
        // The last pass changed nothing; when it made an empty D_t, neither did the one before it.
        k -= !st.c_list && st.n_cur == 0u ? 2u : 1u;
    }
    if (kBatch && a.img_k && still)
        for (int i = tid; i < a.nimg; i += kListThreads)
            if (__ldcg(a.img_n + i) != 0) a.img_k[i] = k;
    if (tid == 0) {
        ctrl->executed += (still ? k : st.k) - k0;
        ctrl->k = k;
        if (!still) ctrl->converged = 1u;
        ctrl->aux = 3u - st.cur - (3u - s_cur - s_aux);  // the other canvas of the pair
        ctrl->cur = st.cur;
        ctrl->work_launches += 1u;
    }
}

namespace {

template <int B, bool kBatch>
cudaError_t launch_loop_b(const PassArgs& a, int sms, cudaStream_t s) {
    int per_sm = 0;
    cudaError_t e =
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, list_loop_kernel<B, kBatch>, kListThreads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    unsigned grid = (unsigned)(sms * (per_sm < 2 ? per_sm : 2));
    if (a.list_ctas > 0 && (unsigned)a.list_ctas < grid) grid = (unsigned)a.list_ctas;
    // A cooperative launch (all CTAs co-resident), in the form that stream
    // capture into a CUDA graph accepts.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kListThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, list_loop_kernel<B, kBatch>, a);
}

template <int B>
cudaError_t launch_loop(const PassArgs& a, int sms, cudaStream_t s) {
    return a.nimg > 1 ? launch_loop_b<B, true>(a, sms, s) : launch_loop_b<B, false>(a, sms, s);
}

}  // namespace

cudaError_t launch_list(int beta, const PassArgs& a, int sms, cudaStream_t s) {
    switch (beta) {
        case 1: return launch_loop<1>(a, sms, s);
        case 2: return launch_loop<2>(a, sms, s);
        case 3: return launch_loop<3>(a, sms, s);
        case 4: return launch_loop<4>(a, sms, s);
        case 5: return launch_loop<5>(a, sms, s);
        case 6: return launch_loop<6>(a, sms, s);
        case 7: return launch_loop<7>(a, sms, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace hg
