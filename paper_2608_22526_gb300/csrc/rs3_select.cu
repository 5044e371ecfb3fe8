// rs3_select.cu -- read-side keep-set K_r (Sec. 3.1: Eq. 1, 2, 4, 5) and the
// write keep-set K_w (Sec. 3.2: Eq. 8), integer-exact.
//
// k_select  the whole selection in one launch: a thread-block cluster of KC
//           CTAs per unit (per group in union mode).  Calls of wide rows, of many
//           objects on one grid or of large unions take three launches through
//           the workspace instead (below; three_launches() draws the line).
//   1. Every CTA turns the unit's mask into bit words (a ballot per 32 cells of
//      a row), updates the tracker (Eq. 4) and dilates: funnel-shifted words
//      along the rows, ORs over rows.  The prior is a bit mask in shared memory.
//      Union mode: the CTAs share the group's units and OR their priors through
//      DSMEM.
//   2. Its cells are listed in ascending order (popc prefix sums); if they are
//      at most k they are the keep-set and no energy is needed.
//   3. Each CTA computes the canonical fp32 ||z||^2 of its share of the list
//      (16-byte loads, up to eight rows in flight per warp, four rows sharing
//      the shuffles of their sums) and stores the keys into the first CTA's
//      shared memory.
//   4. The first CTA finds the k-th largest key with a histogram of 2048 equal
//      bins over the keys' range (energies share their leading bits, which puts
//      a radix pass's keys into a few bins).  A bin of at most 32 keys is
//      ranked by a warp, a fuller one is divided again.  Then it writes the
//      kept cells in ascending order (block scan); in union mode every CTA of the
//      cluster writes some of the group's units.
// Bound by latency and, in one CTA per SM, by instruction issue: 512 threads
// and no divisions in the loops, where 1024 threads took 30 000 cycles.
// One object of 64 x 64 cells and 256 channels takes 7.4 us in a graph of a whole
// sequence's selections, eight 12.5 us, and 16 streams x 3 objects of 96 x 96 20.0 us
// per call (7.3 us at the copy rate); 20.3, 25.9 and 59 us as three launches that
// passed the priors and the energies through global memory.
#include "rs3_cluster.cuh"
#include "rs3_internal.cuh"

#include <algorithm>
#include <climits>
#include <cmath>

#define RS3_NOALLOC_LIMIT (8u << 20)    // largest workspace rs3_select_queries_noalloc stands in for

namespace {

enum { PMODE_EMPTY = 0, PMODE_MASK = 1, PMODE_BOX = 2 };

// ---------------------------------------------------------------------------
// canonical fp32 ||z||^2 (Eq. 5): eight channels of one lane's partial sum
// ---------------------------------------------------------------------------
template <typename T> struct Chunk8;
template <> struct Chunk8<float> {
    float4 a, b;
    __device__ __forceinline__ void load(const float *p)
    {
        a = __ldg(reinterpret_cast<const float4 *>(p));
        b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    }
    __device__ __forceinline__ float add(float s) const
    {
        s = __fmaf_rn(a.x, a.x, s); s = __fmaf_rn(a.y, a.y, s);
        s = __fmaf_rn(a.z, a.z, s); s = __fmaf_rn(a.w, a.w, s);
        s = __fmaf_rn(b.x, b.x, s); s = __fmaf_rn(b.y, b.y, s);
        s = __fmaf_rn(b.z, b.z, s); s = __fmaf_rn(b.w, b.w, s);
        return s;
    }
};
template <> struct Chunk8<uint16_t> {
    uint4 w;
    __device__ __forceinline__ void load(const uint16_t *p) { w = __ldg(reinterpret_cast<const uint4 *>(p)); }
    __device__ __forceinline__ float add(float s) const
    {
        const uint32_t v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float lo = __uint_as_float(v[k] << 16);
            const float hi = __uint_as_float(v[k] & 0xffff0000u);
            s = __fmaf_rn(lo, lo, s);
            s = __fmaf_rn(hi, hi, s);
        }
        return s;
    }
};

// Exclusive block scan of one 32-bit value per thread (values sum < 2^32).
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t &total)
{
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    const int nw = blockDim.x >> 5;
    if (warp == 0) {
        uint32_t x = lane < nw ? s_warp[lane] : 0u;
        uint32_t xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += t;
        }
        if (lane < nw) s_warp[lane] = xi - x;    // exclusive warp offsets
        if (lane == nw - 1) s_total = xi;
    }
    __syncthreads();
    const uint32_t off = s_warp[warp] + (incl - v);
    total = s_total;
    __syncthreads();
    return off;
}

// ---------------------------------------------------------------------------
// k_select
// ---------------------------------------------------------------------------
constexpr int SEL_THREADS = 512, SEL_WARPS = SEL_THREADS / 32;
constexpr int SEL_BINS = 2048;

// Shared memory of a CTA (byte offsets).  The grid's bit words are row by row,
// WW = ceil(n / 32) words each.
struct SelSmem {
    uint32_t prior;      // prior bits; then the histogram
    uint32_t a;          // mask bits and the dilation's first buffer; then the keys
    uint32_t b;          // the dilation's second buffer; then the words' offsets
    uint32_t list;       // uint16: the prior's cells, ascending
    uint32_t total;
};

__host__ __device__ inline SelSmem sel_smem(int m, int n)
{
    const uint32_t mn = (uint32_t)m * n, words = (uint32_t)m * ((n + 31) / 32);
    const auto top = [](uint32_t x, uint32_t y) { return ((x > y ? x : y) + 15u) & ~15u; };
    SelSmem s;
    s.prior = 0;
    s.a = s.prior + top(words * 4, SEL_BINS * 4);
    s.b = s.a + top(words * 4, mn * 4);
    s.list = s.b + top(words * 4, 0);
    s.total = s.list + top(mn * 2, 0);
    return s;
}

// The words threadIdx.x, + SEL_THREADS, ... of the grid's rows of WW words, with
// one division for all of a thread's walks.
struct WordWalk {
    int y0, k0, dy, dk, WW;
    __device__ explicit WordWalk(int ww) : WW(ww)
    {
        y0 = (int)threadIdx.x / ww;
        k0 = (int)threadIdx.x - y0 * ww;
        dy = SEL_THREADS / ww;
        dk = SEL_THREADS - dy * ww;
    }
    template <typename F>
    __device__ __forceinline__ void each(int words, F f) const
    {
        int y = y0, k = k0;
        for (int w = threadIdx.x; w < words; w += SEL_THREADS) {
            f(w, y, k);
            y += dy;
            k += dk;
            if (k >= WW) { k -= WW; ++y; }
        }
    }
};

// A mask's cells as bits of consecutive words, F[i / 32]: a warp's lanes read 32
// adjacent cells, whatever the grid's shape, eight words at a time.
__device__ __forceinline__ void flat_bits(const uint8_t *__restrict__ M, int mn, uint32_t *F)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nf = (mn + 31) >> 5;
    for (int w0 = warp; w0 < nf; w0 += 8 * SEL_WARPS) {
        uint8_t v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int i = 32 * (w0 + q * SEL_WARPS) + lane;
            v[q] = i < mn ? __ldg(M + i) : (uint8_t)0;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint32_t x = __ballot_sync(0xffffffffu, v[q] != 0);
            if (lane == 0 && w0 + q * SEL_WARPS < nf) F[w0 + q * SEL_WARPS] = x;
        }
    }
}

// Word k of row y from them.
__device__ __forceinline__ uint32_t row_word(const uint32_t *F, int nf, int n, int y, int k)
{
    const int i = y * n + 32 * k, w = i >> 5, left = n - 32 * k;
    const uint32_t x = __funnelshift_r(F[w], w + 1 < nf ? F[w + 1] : 0u, i & 31);
    return left < 32 ? x & ((1u << left) - 1u) : x;
}

// Chebyshev dilation of bit words by r: along the rows, by at most 31 cells (a
// neighbouring word) at a time, between the buffers a and b; returns the one
// that holds the result ...
__device__ __forceinline__ uint32_t *dilate_rows(uint32_t *a, uint32_t *b, int words, int n, int r, const WordWalk &walk)
{
    const int WW = walk.WW;
    const uint32_t last = n & 31 ? (1u << (n & 31)) - 1u : 0xffffffffu;   // cells of a row's last word
    uint32_t *from = a, *to = b;
    // (beyond the row's length every cell of a row with a set one is set)
    for (int left = min(r, n); left > 0; left -= 31) {
        const int step = min(left, 31);
        walk.each(words, [&](int w, int, int k) {
            const uint32_t x = from[w], pv = k > 0 ? from[w - 1] : 0u, nx = k < WW - 1 ? from[w + 1] : 0u;
            uint32_t o = x;
            for (int d = 1; d <= step; ++d) o |= __funnelshift_r(x, nx, d) | __funnelshift_l(pv, x, d);
            to[w] = k == WW - 1 ? o & last : o;
        });
        __syncthreads();
        uint32_t *tmp = from;
        from = to;
        to = tmp;
    }
    return from;
}

// ... and over the rows: word w of row y.
__device__ __forceinline__ uint32_t column_or(const uint32_t *from, int w, int y, int m, int r, int WW)
{
    const int up = min(r, y), down = min(r, m - 1 - y);
    uint32_t o = 0u;
#pragma unroll 4
    for (int d = -up; d <= down; ++d) o |= from[w + d * WW];
    return o;
}

// The prior of one unit ORed into P (words of WW per row), with `a` and `b` as
// scratch; thread 0 gets the unit's new tracker state in t.  Every thread of
// the CTA calls it.
__device__ void unit_prior(const uint8_t *__restrict__ M, int m, int n, const WordWalk &walk,
                           const rs3_track *__restrict__ track, int r_s, int c, int bbox_mode, uint32_t *P,
                           uint32_t *a, uint32_t *b, rs3_track &t)
{
    __shared__ int s_box[4][SEL_WARPS];
    __shared__ int s_mode, s_r, s_b[4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int WW = walk.WW, words = m * WW;
    if (threadIdx.x == 0) t = *track;
    int y0 = INT_MAX, x0 = INT_MAX, y1 = -1, x1 = -1;
    flat_bits(M, m * n, b);
    __syncthreads();
    walk.each(words, [&](int w, int y, int k) {
        const uint32_t x = row_word(b, (m * n + 31) >> 5, n, y, k);
        a[w] = x;
        if (x) {
            y0 = min(y0, y);
            y1 = max(y1, y);
            x0 = min(x0, 32 * k + __ffs(x) - 1);
            x1 = max(x1, 32 * k + 31 - __clz(x));
        }
    });
    y0 = __reduce_min_sync(0xffffffffu, y0);
    x0 = __reduce_min_sync(0xffffffffu, x0);
    y1 = __reduce_max_sync(0xffffffffu, y1);
    x1 = __reduce_max_sync(0xffffffffu, x1);
    if (lane == 0) { s_box[0][warp] = y0; s_box[1][warp] = x0; s_box[2][warp] = y1; s_box[3][warp] = x1; }
    __syncthreads();
    if (warp == 0) {
        const int q = lane < SEL_WARPS ? lane : 0;
        y0 = __reduce_min_sync(0xffffffffu, s_box[0][q]);
        x0 = __reduce_min_sync(0xffffffffu, s_box[1][q]);
        y1 = __reduce_max_sync(0xffffffffu, s_box[2][q]);
        x1 = __reduce_max_sync(0xffffffffu, s_box[3][q]);
        if (lane == 0) {
            int mode, r = 0;
            if (y1 >= 0) {                              // non-empty mask (Eq. 1, 2)
                t.y0 = y0; t.x0 = x0; t.y1 = y1; t.x1 = x1;
                t.valid = 1;
                t.streak = 0;
                mode = bbox_mode ? PMODE_BOX : PMODE_MASK;
                r = r_s;
            } else {                                    // empty: streak-counted fallback (Eq. 4)
                if (t.streak < 0x3fffffff) t.streak += 1;
                mode = t.valid ? PMODE_BOX : PMODE_EMPTY;
                if (t.valid) r = r_s + min(t.streak, c);
            }
            s_mode = mode;
            s_r = r;
            s_b[0] = t.y0; s_b[1] = t.x0; s_b[2] = t.y1; s_b[3] = t.x1;
        }
    }
    __syncthreads();
    const int mode = s_mode, r = s_r;
    if (mode == PMODE_MASK) {
        const uint32_t *from = dilate_rows(a, b, words, n, r, walk);
        walk.each(words, [&](int w, int y, int) { P[w] |= column_or(from, w, y, m, r, WW); });
    } else if (mode == PMODE_BOX) {
        const int by0 = s_b[0] - r, bx0 = max(s_b[1] - r, 0), by1 = s_b[2] + r, bx1 = min(s_b[3] + r, n - 1);
        walk.each(words, [&](int w, int y, int k) {
            const int lo = max(bx0 - 32 * k, 0), hi = min(bx1 - 32 * k, 31);    // set bits lo .. hi of the word
            if (y >= by0 && y <= by1 && lo <= hi) P[w] |= (0xffffffffu << lo) & (0xffffffffu >> (31 - hi));
        });
    }
    __syncthreads();
}

// Energies of list entries j0 + warp + SEL_WARPS q, q < UN (a row per warp and
// q: 32 partial sums), into the keys at `key0` of the cluster's first CTA (or
// `keys`).  The 32 partials of four rows are added in the canonical order
// s[l] + s[l + 16], + 8, ...: after the exchange over 16 lanes each half warp
// holds one row of a pair, after the one over 8 each quarter a row of four.
template <typename T, int UN>
struct Energies {
    float s[UN];
    __device__ __forceinline__ void load(const T *zg, const uint16_t *list, uint32_t j0, uint32_t hi, int C)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nchunk = C >> 3;
        const T *row[UN];
#pragma unroll
        for (int q = 0; q < UN; ++q) {
            const uint32_t j = j0 + q * SEL_WARPS + warp;
            row[q] = zg + (size_t)list[min(j, hi - 1u)] * C;
            s[q] = 0.f;
        }
        for (int ch = lane; ch < nchunk; ch += 32) {
            Chunk8<T> x[UN];
#pragma unroll
            for (int q = 0; q < UN; ++q) x[q].load(row[q] + ch * 8);
#pragma unroll
            for (int q = 0; q < UN; ++q) s[q] = x[q].add(s[q]);
        }
    }
    __device__ __forceinline__ void store(uint32_t *keys, uint32_t key0, bool remote, uint32_t j0, uint32_t hi) const
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const bool h16 = lane & 16, h8 = lane & 8;
#pragma unroll
        for (int q = 0; q < UN; q += 4) {
            const float a = (h16 ? s[q + 1] : s[q]) + __shfl_xor_sync(0xffffffffu, h16 ? s[q] : s[q + 1], 16);
            const float b = (h16 ? s[q + 3] : s[q + 2]) + __shfl_xor_sync(0xffffffffu, h16 ? s[q + 2] : s[q + 3], 16);
            float r = (h8 ? b : a) + __shfl_xor_sync(0xffffffffu, h8 ? a : b, 8);
            r = r + __shfl_xor_sync(0xffffffffu, r, 4);
            r = r + __shfl_xor_sync(0xffffffffu, r, 2);
            r = r + __shfl_xor_sync(0xffffffffu, r, 1);
            const uint32_t j = j0 + (q + (h16 ? 1 : 0) + (h8 ? 2 : 0)) * SEL_WARPS + warp;
            if ((lane & 7) == 0 && j < hi) {
                if (remote) dsmem_st_u32(key0 + 4 * j, __float_as_uint(r));
                else keys[j] = __float_as_uint(r);
            }
        }
    }
};

// The keys of list entries [lo, hi) by a CTA; before() runs ahead of the first
// store.  lpr lanes share a row: 32, or fewer that hold one chunk each.
template <typename T, typename F>
__device__ __forceinline__ void energies(const T *zg, const uint16_t *list, uint32_t lo, uint32_t hi, int C, int lpr,
                                         uint32_t *keys, uint32_t key0, bool remote, F before)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lpr == 32) {
        constexpr int UN = sizeof(T) == 2 ? 8 : 4;
        for (uint32_t j0 = lo; j0 < hi; j0 += UN * SEL_WARPS) {
            Energies<T, UN> e;
            e.load(zg, list, j0, hi, C);
            before();
            e.store(keys, key0, remote, j0, hi);
        }
        return;
    }
    const int nchunk = C >> 3, rpw = 32 / lpr, sub = lane / lpr, l = lane % lpr;
    constexpr int UN = 4;
    for (uint32_t j0 = lo; j0 < hi; j0 += UN * SEL_WARPS * rpw) {
        Chunk8<T> x[UN];
        float s[UN];
#pragma unroll
        for (int q = 0; q < UN; ++q) {
            const uint32_t j = j0 + (q * SEL_WARPS + warp) * rpw + sub;
            if (l < nchunk) x[q].load(zg + (size_t)list[min(j, hi - 1u)] * C + l * 8);
        }
#pragma unroll
        for (int q = 0; q < UN; ++q) {
            s[q] = l < nchunk ? x[q].add(0.f) : 0.f;
            for (int w = lpr >> 1; w >= 1; w >>= 1) s[q] = s[q] + __shfl_xor_sync(0xffffffffu, s[q], w);
        }
        before();
#pragma unroll
        for (int q = 0; q < UN; ++q) {
            const uint32_t j = j0 + (q * SEL_WARPS + warp) * rpw + sub;
            if (j < hi && l == 0) {
                if (remote) dsmem_st_u32(key0 + 4 * j, __float_as_uint(s[q]));
                else keys[j] = __float_as_uint(s[q]);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// ranking (by a whole CTA)
// ---------------------------------------------------------------------------
// Which keys are kept: those >= from, and the first `want` of those == equal.
// `all`: every one (no key was needed).
struct Kept {
    uint32_t from = 0u, equal = 0xffffffffu, want = 0u;
    bool all = true;
};

// The k largest of nP keys (0 < k < nP), `hist` SEL_BINS words of scratch.
__device__ __forceinline__ Kept top_keys(const uint32_t *keys, uint32_t nP, uint32_t k, uint32_t *hist)
{
    __shared__ uint32_t s_bin, s_rem, s_cnt, s_ncand, s_cand[32], s_mm[2][SEL_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Kept r;
    r.all = false;
    if (threadIdx.x == 0) s_ncand = 0u;
    for (int b = threadIdx.x; b < SEL_BINS; b += SEL_THREADS) hist[b] = 0;
    __syncthreads();                                     // (and the keys)
    // the range of the keys
    uint32_t mi = 0xffffffffu, ma = 0u;
    for (uint32_t j = threadIdx.x; j < nP; j += SEL_THREADS) {
        mi = min(mi, keys[j]);
        ma = max(ma, keys[j]);
    }
    mi = __reduce_min_sync(0xffffffffu, mi);
    ma = __reduce_max_sync(0xffffffffu, ma);
    if (lane == 0) { s_mm[0][warp] = mi; s_mm[1][warp] = ma; }
    __syncthreads();
    mi = __reduce_min_sync(0xffffffffu, s_mm[0][lane % SEL_WARPS]);
    ma = __reduce_max_sync(0xffffffffu, s_mm[1][lane % SEL_WARPS]);
    // keys of bin b of a pass lie in [base + (b << shift), base + ((b + 1) <<
    // shift)); want: how many of the range's largest keys are kept
    uint32_t base = mi, span = ma - mi;
    r.want = k;
    int shift = max(0, 32 - __clz(span | 1u) - 11);
    for (;;) {
        for (uint32_t j = threadIdx.x; j < nP; j += SEL_THREADS) {
            const uint32_t d = keys[j] - base;           // wraps past every span for keys below base
            if (d <= span) atomicAdd(&hist[d >> shift], 1u);
        }
        __syncthreads();
        // thread t takes four bins, from the top
        const uint4 h = reinterpret_cast<const uint4 *>(hist)[SEL_BINS / 4 - 1 - threadIdx.x];
        uint32_t tot, above = block_excl_scan((h.x + h.y) + (h.z + h.w), tot);
        if (above < r.want && r.want <= above + (h.x + h.y) + (h.z + h.w)) {
            const uint32_t x[4] = {h.w, h.z, h.y, h.x};
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                if (above < r.want && r.want <= above + x[b]) {
                    s_bin = SEL_BINS - 1 - 4 * threadIdx.x - b;
                    s_rem = r.want - above;
                    s_cnt = x[b];
                }
                above += x[b];
            }
        }
        __syncthreads();
        base += s_bin << shift;
        r.want = s_rem;
        span = (1u << shift) - 1u;
        if (s_cnt == r.want) {                           // the whole bin is kept
            r.from = base;
            r.want = 0u;
            return r;
        }
        if (shift == 0) {                                // a bin of equal keys
            r.from = base + 1u;
            r.equal = base;
            return r;
        }
        if (s_cnt <= 32u) {                              // a warp ranks them (each for itself)
            for (uint32_t j = threadIdx.x; j < nP; j += SEL_THREADS)
                if (keys[j] - base <= span) s_cand[atomicAdd(&s_ncand, 1u)] = keys[j];
            __syncthreads();
            const int nc = (int)s_cnt;
            const uint32_t x = s_cand[lane < nc ? lane : 0];
            uint32_t gt = 0, ge = 0;
            for (int i = 0; i < nc; ++i) {
                const uint32_t y = __shfl_sync(0xffffffffu, x, i);
                gt += y > x ? 1u : 0u;
                ge += y >= x ? 1u : 0u;
            }
            const int at = __ffs(__ballot_sync(0xffffffffu, lane < nc && gt < r.want && r.want <= ge)) - 1;
            r.equal = __shfl_sync(0xffffffffu, x, at);
            r.from = r.equal + 1u;
            r.want -= __shfl_sync(0xffffffffu, gt, at);
            return r;
        }
        shift = max(0, shift - 11);
        for (int b = threadIdx.x; b < SEL_BINS; b += SEL_THREADS) hist[b] = 0;
        __syncthreads();
    }
}

// Where the kept cells go.  Each thread a run of the list; a kept cell's place is
// the number of kept larger keys before it and of equal ones, of which the first
// `want` are kept.
struct Place {
    uint32_t j0, j1, off;
    __device__ __forceinline__ Place(const uint32_t *keys, uint32_t nP, const Kept &r)
    {
        const uint32_t per = (nP + SEL_THREADS - 1) / SEL_THREADS;
        j0 = threadIdx.x * per;
        j1 = min(j0 + per, nP);
        off = 0u;
        if (r.all) return;
        uint32_t mine = 0, tot;
        for (uint32_t j = j0; j < j1; ++j) mine += (keys[j] >= r.from ? 0x10000u : 0u) + (keys[j] == r.equal ? 1u : 0u);
        off = block_excl_scan(mine, tot);
    }
    // the kept cells of the list in order, into `out`, which may lie over the keys
    __device__ __forceinline__ void compact(const uint32_t *keys, const uint16_t *list, const Kept &r, uint16_t *out) const
    {
        uint32_t at = (off >> 16) + min(off & 0xffffu, r.want), eq = off & 0xffffu, flags = 0u;
        for (uint32_t j = j0; j < j1; ++j) {             // at most 32: a run of 16384 / SEL_THREADS cells
            const uint32_t key = keys[j];
            const bool is_eq = key == r.equal;
            if (key >= r.from || (is_eq && eq < r.want)) flags |= 1u << (j - j0);
            eq += is_eq ? 1u : 0u;
        }
        __syncthreads();
        for (; flags; flags &= flags - 1) out[at++] = list[j0 + __ffs(flags) - 1];
        __syncthreads();
    }
    // one unit's row of the output and its count
    __device__ __forceinline__ void emit(const uint32_t *keys, const uint16_t *list, const Kept &r, uint32_t n_kept, int32_t *out,
                         int32_t *count) const
    {
        if (r.all) {
            for (uint32_t j = threadIdx.x; j < n_kept; j += SEL_THREADS) out[j] = list[j];
        } else {
            uint32_t gt = off >> 16, eq = off & 0xffffu;
            for (uint32_t j = j0; j < j1; ++j) {
                const uint32_t key = keys[j];
                const bool is_eq = key == r.equal;
                if (key >= r.from || (is_eq && eq < r.want)) out[gt + min(eq, r.want)] = list[j];
                gt += key >= r.from ? 1u : 0u;
                eq += is_eq ? 1u : 0u;
            }
        }
        if (threadIdx.x == 0) *count = (int32_t)n_kept;
    }
};

// (bf16: eight rows' loads in flight take 64 registers; left to itself the compiler
// stops at 54 and waits in between: 16 x 3 objects of 96 x 96 23.1 us, 21.0 so)
template <typename T>
__global__ void __launch_bounds__(SEL_THREADS, sizeof(T) == 2 ? 2 : 1)
k_select(const T *__restrict__ z, const uint8_t *__restrict__ masks, int m, int n, int C, int lpr,
         const int32_t *__restrict__ unit_group, int G, int U, rs3_track *__restrict__ track, int r_s, int c,
         int bbox_mode, int union_mode, int k, int KC, int32_t *__restrict__ idx, int32_t *__restrict__ count,
         int32_t *status)
{
    pdl_wait();
    extern __shared__ __align__(16) uint8_t sel_raw[];
    const SelSmem S = sel_smem(m, n);
    uint32_t *P = reinterpret_cast<uint32_t *>(sel_raw + S.prior), *hist = P;
    uint32_t *A = reinterpret_cast<uint32_t *>(sel_raw + S.a), *keys = A;
    uint32_t *B = reinterpret_cast<uint32_t *>(sel_raw + S.b), *pref = B;
    uint16_t *list = reinterpret_cast<uint16_t *>(sel_raw + S.list);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int u = blockIdx.x / KC;
    const uint32_t rank = KC > 1 ? cluster_rank() : 0u;
    const int mn = m * n, WW = (n + 31) >> 5, words = m * WW;
    if (union_mode) {
        // a cluster per group: its first unit, if it has one
        __shared__ int s_first;
        const int group = u;
        if (threadIdx.x == 0) s_first = U;
        __syncthreads();
        for (int v = threadIdx.x; v < U; v += SEL_THREADS) {
            const int gv = unit_group[v];
            if (gv == group) atomicMin(&s_first, v);
            if ((gv < 0 || gv >= G) && group == 0 && rank == 0) {
                latch_status(status, RS3_EINVAL);
                count[v] = 0;
            }
        }
        __syncthreads();
        u = s_first;
        if (u >= U) return;                              // uniform over the cluster
    }
    const int g = unit_group[u];
    if (g < 0 || g >= G) {                               // uniform over the cluster
        if (rank == 0 && threadIdx.x == 0) {
            latch_status(status, RS3_EINVAL);
            count[u] = 0;
        }
        return;
    }
    const WordWalk walk(WW);
    for (int w = threadIdx.x; w < words; w += SEL_THREADS) P[w] = 0u;
    rs3_track tr = {};
    if (!union_mode) {
        // (P is read again only after this call's first barrier)
        unit_prior(masks + (size_t)u * mn, m, n, walk, track + u, r_s, c, bbox_mode, P, A, B, tr);
    } else {
        __syncthreads();
        uint32_t seen = 0;
        for (int v0 = u; v0 < U; v0 += 32) {             // members in order; rank r takes r, r + KC, ...
            uint32_t in = __ballot_sync(0xffffffffu, v0 + lane < U && unit_group[min(v0 + lane, U - 1)] == g);
            for (; in; in &= in - 1, ++seen) {
                if (seen % (uint32_t)KC != rank) continue;
                const int v = v0 + __ffs(in) - 1;
                unit_prior(masks + (size_t)v * mn, m, n, walk, track + v, r_s, c, bbox_mode, P, A, B, tr);
                if (threadIdx.x == 0) track[v] = tr;     // no other CTA reads it
            }
        }
        if (KC > 1) {
            cluster_arrive();
            cluster_wait();
            for (int w = threadIdx.x; w < words; w += SEL_THREADS) {
                uint32_t o = P[w];
                for (int q = 0; q < KC; ++q) o |= dsmem_ld_u32(dsmem_addr(P + w, (uint32_t)q));
                A[w] = o;
            }
            cluster_arrive();
            cluster_wait();                              // every CTA has read this one's
            for (int w = threadIdx.x; w < words; w += SEL_THREADS) P[w] = A[w];
            __syncthreads();
        }
    }

    // the prior's cells in ascending order
    uint32_t nP;
    {
        const int per = (words + SEL_THREADS - 1) / SEL_THREADS, w0 = threadIdx.x * per;
        uint32_t own = 0;
        for (int w = w0; w < min(w0 + per, words); ++w) own += __popc(P[w]);
        uint32_t off = block_excl_scan(own, nP);
        for (int w = w0; w < min(w0 + per, words); ++w) {
            pref[w] = off;
            off += __popc(P[w]);
        }
    }
    __syncthreads();
    const uint32_t below = (1u << lane) - 1u;
    if (n >= 8) {                                        // a lane per bit, or, in narrow rows, a thread per row
        for (int y = warp; y < m; y += SEL_WARPS)
            for (int k = 0; k < WW; ++k) {
                const uint32_t bits = P[y * WW + k];
                if (bits >> lane & 1u) list[pref[y * WW + k] + __popc(bits & below)] = (uint16_t)(y * n + 32 * k + lane);
            }
    } else {
        for (int y = threadIdx.x; y < m; y += SEL_THREADS) {
            uint32_t at = pref[y];
            for (uint32_t bits = P[y]; bits; bits &= bits - 1) list[at++] = (uint16_t)(y * n + __ffs(bits) - 1);
        }
    }
    const bool keep_all = nP <= (uint32_t)k;
    const uint32_t n_kept = keep_all ? nP : (uint32_t)k;
    __syncthreads();
    // the keys may be written once the first CTA no longer needs its bit words;
    // it writes the tracker once every CTA has read the old one
    if (KC > 1) cluster_arrive();
    if (!keep_all && k > 0) {
        const uint32_t share = (nP + KC - 1) / KC, lo = min(rank * share, nP), hi = min(lo + share, nP);
        const uint32_t key0 = KC > 1 ? dsmem_addr(keys, 0u) : 0u;
        const T *zg = z + (size_t)g * mn * C;
        bool waited = KC == 1;
        energies<T>(zg, list, lo, hi, C, lpr, keys, key0, KC > 1, [&]() {
            if (!waited) cluster_wait();
            waited = true;
        });
        if (!waited) cluster_wait();
        if (KC > 1) {
            cluster_arrive();
            cluster_wait();
        }
    } else if (KC > 1) {
        cluster_wait();
    }
    const bool ranked = !keep_all && k > 0;
    if (!union_mode) {
        if (rank != 0) return;
        if (threadIdx.x == 0) track[u] = tr;
        const Kept kept = ranked ? top_keys(keys, nP, (uint32_t)k, hist) : Kept{};
        const Place place(keys, nP, kept);
        place.emit(keys, list, kept, n_kept, idx + (size_t)u * k, count + u);
        return;
    }
    // union mode: the first CTA ranks, every CTA writes the group's units in turn
    const uint16_t *kept_list = list;
    if (ranked) {
        if (rank == 0) {
            const Kept kept = top_keys(keys, nP, (uint32_t)k, hist);
            const Place place(keys, nP, kept);
            place.compact(keys, list, kept, reinterpret_cast<uint16_t *>(keys));
        }
        if (KC > 1) {
            cluster_arrive();
            cluster_wait();
            if (rank != 0)
                for (uint32_t i = threadIdx.x; i < (n_kept + 1) / 2; i += SEL_THREADS)
                    keys[i] = dsmem_ld_u32(dsmem_addr(keys + i, 0u));
            cluster_arrive();
        }
        __syncthreads();
        kept_list = reinterpret_cast<const uint16_t *>(keys);
    }
    uint32_t seen = 0;
    for (int v0 = u; v0 < U; v0 += 32) {
        uint32_t in = __ballot_sync(0xffffffffu, v0 + lane < U && unit_group[min(v0 + lane, U - 1)] == g);
        for (; in; in &= in - 1, ++seen) {
            if (seen % (uint32_t)KC != rank) continue;
            const int v = v0 + __ffs(in) - 1;
            int32_t *out = idx + (size_t)v * k;
            for (uint32_t j = threadIdx.x; j < n_kept; j += SEL_THREADS) out[j] = kept_list[j];
            if (threadIdx.x == 0) count[v] = (int32_t)n_kept;
        }
    }
    if (ranked && KC > 1) cluster_wait();                // every CTA has read the first one's list
}

// ---------------------------------------------------------------------------
// The selection in three launches, through the workspace, for calls whose rows are
// too much for the few SMs that a unit's cluster has, or whose objects share them:
//   k_prior   a CTA per unit: tracker and prior; bit i of a unit's (or, in union
//             mode, the group's) cells, and the cells that the group needs
//   k_energy  the energies of the needed cells, over all SMs
//   k_rank    a CTA per unit: lists, ranks and writes
// ---------------------------------------------------------------------------
struct SelWs {           // in the workspace; nf = ceil(mn / 32) words hold a bit per cell
    uint32_t *need;      // [G][nf]
    uint32_t *prior;     // [U][nf]
    uint32_t *energy;    // [G][mn] bits of the fp32 energies
};

__global__ void __launch_bounds__(SEL_THREADS)
k_prior(const uint8_t *__restrict__ masks, int m, int n, const int32_t *__restrict__ unit_group, int G,
        rs3_track *__restrict__ track, int r_s, int c, int bbox_mode, int union_mode, SelWs ws, int32_t *status)
{
    pdl_wait();
    extern __shared__ __align__(16) uint8_t sel_raw[];
    const int mn = m * n, WW = (n + 31) >> 5, words = m * WW, nf = (mn + 31) >> 5, u = blockIdx.x, g = unit_group[u];
    if (g < 0 || g >= G) {                               // k_rank writes its count
        if (threadIdx.x == 0) latch_status(status, RS3_EINVAL);
        return;
    }
    uint32_t *P = reinterpret_cast<uint32_t *>(sel_raw), *A = P + words, *B = A + words, *F = B + words;
    for (int w = threadIdx.x; w < words; w += SEL_THREADS) P[w] = 0u;
    for (int w = threadIdx.x; w < nf; w += SEL_THREADS) F[w] = 0u;
    const WordWalk walk(WW);
    rs3_track tr = {};
    unit_prior(masks + (size_t)u * mn, m, n, walk, track + u, r_s, c, bbox_mode, P, A, B, tr);
    if (threadIdx.x == 0) track[u] = tr;
    // words of a row -> bits of consecutive cells
    walk.each(words, [&](int w, int y, int k) {
        const uint32_t x = P[w];
        const int i = y * n + 32 * k, sh = i & 31;
        if (x == 0u) return;
        atomicOr(&F[i >> 5], x << sh);
        if (sh && x >> (32 - sh)) atomicOr(&F[(i >> 5) + 1], x >> (32 - sh));
    });
    __syncthreads();
    for (int w = threadIdx.x; w < nf; w += SEL_THREADS) {
        if (!union_mode) ws.prior[(size_t)u * nf + w] = F[w];
        if (F[w]) atomicOr(&ws.need[(size_t)g * nf + w], F[w]);
    }
}

// The set cells of words [w0, w0 + nw) in ascending order; every thread of the
// CTA calls it.  Returns their number.
__device__ __forceinline__ uint32_t list_bits(const uint32_t *F, int w0, int nw, uint16_t *list)
{
    const int per = (nw + SEL_THREADS - 1) / SEL_THREADS, a = threadIdx.x * per, b = min(a + per, nw);
    uint32_t own = 0, total;
    for (int w = a; w < b; ++w) own += __popc(F[w0 + w]);
    uint32_t off = block_excl_scan(own, total);
    for (int w = a; w < b; ++w)
        for (uint32_t x = F[w0 + w]; x; x &= x - 1) list[off++] = (uint16_t)(32 * (w0 + w) + __ffs(x) - 1);
    __syncthreads();
    return total;
}

// A warp per row (per 32 / lpr rows of few channels), over all of the groups' rows.
template <typename T>
__global__ void __launch_bounds__(256)
k_energy(const T *__restrict__ z, int G, int mn, int C, int lpr, SelWs ws)
{
    pdl_wait();
    const int nchunk = C >> 3, rpw = 32 / lpr, lane = threadIdx.x & 31, sub = lane / lpr, l = lane % lpr;
    const int nf = (mn + 31) >> 5;
    const long total = (long)G * mn;
    const long wid = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = ((long)gridDim.x * blockDim.x) >> 5;
    for (long base = wid * rpw; base < total; base += nwarps * rpw) {
        const long row = base + sub;
        bool needed = false;
        if (row < total) {
            const int g = (int)(row / mn), i = (int)(row - (long)g * mn);
            needed = (ws.need[(size_t)g * nf + (i >> 5)] >> (i & 31)) & 1u;
        }
        float s = 0.0f;
        if (needed) {
            const T *zr = z + row * (long)C;
            for (int ch = l; ch < nchunk; ch += 32) {
                Chunk8<T> x;
                x.load(zr + ch * 8);
                s = x.add(s);
            }
        }
        for (int w = lpr >> 1; w >= 1; w >>= 1) s = s + __shfl_xor_sync(0xffffffffu, s, w);
        if (needed && l == 0) ws.energy[row] = __float_as_uint(s);
    }
}

// Shared memory: histogram, keys, list.
__global__ void __launch_bounds__(SEL_THREADS)
k_rank(int mn, const int32_t *__restrict__ unit_group, int G, int union_mode, int k, SelWs ws, int32_t *__restrict__ idx,
       int32_t *__restrict__ count)
{
    pdl_wait();
    extern __shared__ __align__(16) uint8_t sel_raw[];
    uint32_t *hist = reinterpret_cast<uint32_t *>(sel_raw), *keys = hist + SEL_BINS;
    uint16_t *list = reinterpret_cast<uint16_t *>(keys + mn);
    const int nf = (mn + 31) >> 5, u = blockIdx.x, g = unit_group[u];
    if (g < 0 || g >= G) {
        if (threadIdx.x == 0) count[u] = 0;
        return;
    }
    const uint32_t nP = list_bits(union_mode ? ws.need + (size_t)g * nf : ws.prior + (size_t)u * nf, 0, nf, list);
    const bool keep_all = nP <= (uint32_t)k;
    if (!keep_all)
        for (uint32_t j = threadIdx.x; j < nP; j += SEL_THREADS) keys[j] = ws.energy[(size_t)g * mn + list[j]];
    const Kept kept = keep_all || k == 0 ? Kept{} : top_keys(keys, nP, (uint32_t)k, hist);
    const Place place(keys, nP, kept);
    place.emit(keys, list, kept, keep_all ? nP : (uint32_t)k, idx + (size_t)u * k, count + u);
}

// ---------------------------------------------------------------------------
// k_write_keepset: Eq. 8 with the 5% / 95% fall-through of Sec. 3.2, a CTA per
// unit on bit words.  64 x 64 cells, radius 24, in a graph: 4.8 us, 12.2 cell by
// cell; union of 48 objects 13.7 us, 46.
// ---------------------------------------------------------------------------
// The union of a group's masks as bits (as flat_bits): four words of eight masks
// in flight per warp.  Every thread of the CTA calls it.
__device__ __forceinline__ void group_bits(const uint8_t *__restrict__ masks, int mn, const int32_t *__restrict__ unit_group,
                                           int U, int g, uint32_t *F)
{
    __shared__ int s_unit[SEL_THREADS], s_n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nf = (mn + 31) >> 5;
    for (int w = threadIdx.x; w < nf; w += SEL_THREADS) F[w] = 0u;
    for (int v0 = 0; v0 < U; v0 += SEL_THREADS) {
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        const int v = v0 + threadIdx.x;
        if (v < U && unit_group[v] == g) s_unit[atomicAdd(&s_n, 1)] = v;     // (in any order)
        __syncthreads();
        const int units = s_n;
        for (int w0 = warp; w0 < nf; w0 += 4 * SEL_WARPS) {
            uint32_t any[4] = {0u, 0u, 0u, 0u};
            for (int j0 = 0; j0 < units; j0 += 8) {
                uint8_t x[8][4];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint8_t *M = masks + (size_t)s_unit[min(j0 + j, units - 1)] * mn;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int i = 32 * (w0 + q * SEL_WARPS) + lane;
                        x[j][q] = i < mn ? __ldg(M + i) : (uint8_t)0;
                    }
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q) any[q] |= x[j][q];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t b = __ballot_sync(0xffffffffu, any[q] != 0u);
                if (lane == 0 && w0 + q * SEL_WARPS < nf) F[w0 + q * SEL_WARPS] |= b;   // always this warp's
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(SEL_THREADS)
k_write_keepset(const uint8_t *__restrict__ seeds, const int32_t *__restrict__ unit_group, int U, int m, int n,
                int D_w, double fall_lo, double fall_hi, int fall_through, int union_mode, uint8_t *__restrict__ kw)
{
    pdl_wait();
    extern __shared__ __align__(16) uint8_t sel_raw[];
    const int mn = m * n, WW = (n + 31) >> 5, words = m * WW, u = blockIdx.x;
    uint32_t *a = reinterpret_cast<uint32_t *>(sel_raw), *b = a + words;
    const WordWalk walk(WW);
    if (union_mode) group_bits(seeds, mn, unit_group, U, unit_group[u], b);
    else flat_bits(seeds + (size_t)u * mn, mn, b);
    __syncthreads();
    walk.each(words, [&](int w, int y, int k) { a[w] = row_word(b, (mn + 31) >> 5, n, y, k); });
    __syncthreads();
    uint32_t own = 0, area;
    for (int w = threadIdx.x; w < words; w += SEL_THREADS) own += __popc(a[w]);
    block_excl_scan(own, area);
    const double frac = (double)area / (double)mn;
    uint8_t *out = kw + (size_t)u * mn;
    if (fall_through && (frac > fall_hi || frac < fall_lo)) {
        for (int i = threadIdx.x; i < mn; i += SEL_THREADS) out[i] = 1;
        return;
    }
    uint32_t *from = dilate_rows(a, b, words, n, D_w, walk), *to = from == a ? b : a;
    walk.each(words, [&](int w, int y, int) { to[w] = column_or(from, w, y, m, D_w, WW); });
    __syncthreads();
    const int dy = SEL_THREADS / n, dx = SEL_THREADS - dy * n;
    int y = (int)threadIdx.x / n, x = (int)threadIdx.x - y * n;
    for (int i = threadIdx.x; i < mn; i += SEL_THREADS) {
        out[i] = (uint8_t)(to[y * WW + (x >> 5)] >> (x & 31) & 1u);
        y += dy;
        x += dx;
        if (x >= n) { x -= n; ++y; }
    }
}

inline int next_pow2(int x)
{
    int p = 1;
    while (p < x) p <<= 1;
    return p;
}

}  // namespace

// ---------------------------------------------------------------------------
// host entry points
// ---------------------------------------------------------------------------
namespace {

// Byte offsets in the workspace of the three-launch selection.  The size is part
// of the ABI; the prior's region holds a byte per cell, of which bits are used.
struct SelectWs {
    size_t prior, energy, total;
};

SelectWs select_ws(int G, int U, int m, int n)
{
    const size_t mn = (size_t)m * n;
    SelectWs w;
    w.prior = align_up((size_t)G * ((mn + 31) / 32) * 4, 256);
    w.energy = align_up(w.prior + (size_t)U * mn, 256);
    w.total = align_up(w.energy + (size_t)G * mn * 4, 256);
    return w;
}

}  // namespace

extern "C" size_t rs3_select_workspace_bytes(int G, int U, int m, int n)
{
    if (G < 1 || U < 1 || m < 1 || n < 1) return 0;
    return select_ws(G, U, m, n).total;
}

namespace {

rs3_status select_check(const void *z, rs3_dtype dtype, int G, int m, int n, int C, const uint8_t *prev_masks,
                        const int32_t *unit_group, int U, const rs3_track *track, const rs3_params *p,
                        const int32_t *idx, const int32_t *count, const int32_t *status)
{
    if (!z || !prev_masks || !unit_group || !track || !p || !idx || !count || !status) return RS3_EINVAL;
    if (dtype != RS3_F32 && dtype != RS3_BF16) return RS3_EINVAL;
    if (G < 1 || U < 1 || m < 1 || n < 1 || C < 8 || (C % 8) != 0) return RS3_EINVAL;
    if ((long)m * n > RS3_MAX_MN || C > 4096) return RS3_EUNSUPPORTED;
    if (!(p->rho >= 0.0 && p->rho <= 1.0) || p->r_s < 0 || p->c < 0) return RS3_EINVAL;
    if (!rs3_aligned16(z)) return RS3_EINVAL;
    return RS3_OK;
}

// Whether three launches are the faster, by what both take when most of the grid
// is in the priors (us on 152 SMs).  One launch: the share of a unit's channels that
// each CTA of its cluster reads, at two CTAs per SM half as fast.  Three: their fixed
// cost, the rows that all SMs walk and the bytes they read.  One object on 64 x 64
// cells: 256 bf16 channels 11.6 us in one launch, 18.4 in three; 2048 channels 42 and
// 20; 16 x 3 objects on 96 x 96, 256 channels 45 and 52; 255 objects of one grid 33
// and 19.  (The memset, prior, energy and select kernels before took 22, 26, 66 and
// 31.)  Where nothing has to be ranked one launch reads no rows, and three cost 12 us
// instead of 5, still less than before.  Union mode: units past a CTA each are
// worked off in turn by a cluster, but side by side in three launches.
bool three_launches(int G, int U, int mn, int C, size_t esz, int union_mode, long clusters, int KC, int n_sm)
{
    if (union_mode && U > (long)G * KC) return true;
    const double share = (double)mn * C / KC, rows = (double)G * mn;
    const double one = 6.0 + 36e-6 * share * std::max(1.0, (double)clusters * KC / n_sm);
    const double three = 16.0 + 0.12e-3 * rows + 0.05e-6 * rows * C * (double)esz;
    return one > three;
}

// The selection: one launch, or three through the workspace (null: one).
rs3_status select_launch(const void *z, rs3_dtype dtype, int G, int m, int n, int C, const uint8_t *prev_masks,
                         const int32_t *unit_group, int U, rs3_track *track, const rs3_params *p, int32_t *idx,
                         int32_t *count, void *workspace, int32_t *status, rs3_stream_t stream)
{
    const int mn = m * n;
    const int64_t k = rs3_kmax(p->rho, (int64_t)mn);
    if (k < 0) return RS3_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // CTAs per cluster: as many as are resident at once (two per SM), up to the
    // portable 8; 48 units of 96 x 96 cells, both then: 20.9 us with 6 each, 22.6 with 4
    const long clusters = p->union_mode ? (G < U ? G : U) : U;
    const int n_sm = rs3_sm_count();
    const int KC = (int)std::min(8l, std::max(1l, 2l * n_sm / clusters));
    const int nchunk = C / 8;
    const int lpr = nchunk >= 32 ? 32 : next_pow2(nchunk);
    cudaError_t e;
    if (workspace && mn >= 4 &&             // (a unit's bits fit its bytes of the workspace)
        three_launches(G, U, mn, C, dtype == RS3_BF16 ? 2 : 4, p->union_mode, clusters, KC, n_sm)) {
        const int nf = (mn + 31) / 32;
        const SelectWs l = select_ws(G, U, m, n);
        uint8_t *b = static_cast<uint8_t *>(workspace);
        const SelWs ws = {reinterpret_cast<uint32_t *>(b), reinterpret_cast<uint32_t *>(b + l.prior),
                          reinterpret_cast<uint32_t *>(b + l.energy)};
        const size_t prior_smem = 4 * (3 * (size_t)m * ((n + 31) / 32) + nf);
        const size_t rank_smem = 4 * SEL_BINS + 6 * (size_t)mn;
        if (rs3_kernel_smem((const void *)k_prior, prior_smem + 1024) != RS3_OK ||      // + its static arrays
            rs3_kernel_smem((const void *)k_rank, rank_smem + 1024) != RS3_OK)
            return RS3_ECUDA;
        if (cudaMemsetAsync(ws.need, 0, (size_t)G * nf * 4, st) != cudaSuccess) return RS3_ECUDA;
        e = launch_pdl(k_prior, dim3(U), dim3(SEL_THREADS), prior_smem, st, prev_masks, m, n, unit_group, G, track, p->r_s,
                       p->c, p->bbox_mode, p->union_mode, ws, status);
        const long warps = ((long)G * mn + 32 / lpr - 1) / (32 / lpr);
        const dim3 grid((unsigned)std::min((warps + 7) / 8, 8l * n_sm));
        if (e == cudaSuccess)
            e = dtype == RS3_BF16 ? launch_pdl(k_energy<uint16_t>, grid, dim3(256), 0, st, static_cast<const uint16_t *>(z),
                                               G, mn, C, lpr, ws)
                                  : launch_pdl(k_energy<float>, grid, dim3(256), 0, st, static_cast<const float *>(z), G, mn,
                                               C, lpr, ws);
        if (e == cudaSuccess)
            e = launch_pdl(k_rank, dim3(U), dim3(SEL_THREADS), rank_smem, st, mn, unit_group, G, p->union_mode, (int)k, ws,
                           idx, count);
        return e == cudaSuccess ? RS3_OK : RS3_ECUDA;
    }
    const size_t smem = sel_smem(m, n).total;
    const void *fn = dtype == RS3_BF16 ? (const void *)k_select<uint16_t> : (const void *)k_select<float>;
    if (rs3_kernel_smem(fn, smem + 1024) != RS3_OK) return RS3_ECUDA;       // + the kernel's static arrays
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((p->union_mode ? G : U) * KC));    // a cluster per group in union mode
    cfg.blockDim = dim3(SEL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = KC;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if (dtype == RS3_BF16)
        e = cudaLaunchKernelEx(&cfg, k_select<uint16_t>, static_cast<const uint16_t *>(z), prev_masks, m, n, C, lpr,
                               unit_group, G, U, track, p->r_s, p->c, p->bbox_mode, p->union_mode, (int)k, KC, idx,
                               count, status);
    else
        e = cudaLaunchKernelEx(&cfg, k_select<float>, static_cast<const float *>(z), prev_masks, m, n, C, lpr,
                               unit_group, G, U, track, p->r_s, p->c, p->bbox_mode, p->union_mode, (int)k, KC, idx,
                               count, status);
    return e == cudaSuccess ? RS3_OK : RS3_ECUDA;
}

}  // namespace

extern "C" rs3_status rs3_select_queries(const void *z, rs3_dtype dtype, int G, int m, int n, int C,
                                         const uint8_t *prev_masks, const int32_t *unit_group,
                                         int U, rs3_track *track, const rs3_params *p,
                                         int32_t *idx, int32_t *count, void *workspace,
                                         size_t workspace_bytes, int32_t *status,
                                         rs3_stream_t stream)
{
    if (!workspace) return RS3_EINVAL;
    const rs3_status s = select_check(z, dtype, G, m, n, C, prev_masks, unit_group, U, track, p, idx, count, status);
    if (s != RS3_OK) return s;
    if (!rs3_aligned16(workspace)) return RS3_EINVAL;
    if (workspace_bytes < rs3_select_workspace_bytes(G, U, m, n)) return RS3_ECAPACITY;
    return select_launch(z, dtype, G, m, n, C, prev_masks, unit_group, U, track, p, idx, count, workspace, status,
                         stream);
}

// rs3_select_queries for callers that cannot allocate device memory: the same
// launch, without the workspace pair.
extern "C" rs3_status rs3_select_queries_noalloc(const void *z, rs3_dtype dtype, int G, int m, int n, int C,
                                                 const uint8_t *prev_masks, const int32_t *unit_group, int U,
                                                 rs3_track *track, const rs3_params *p, int32_t *idx,
                                                 int32_t *count, int32_t *status, rs3_stream_t stream)
{
    const size_t need = rs3_select_workspace_bytes(G, U, m, n);
    if (need == 0) return RS3_EINVAL;
    if (need > RS3_NOALLOC_LIMIT) return RS3_ECAPACITY;
    const rs3_status s = select_check(z, dtype, G, m, n, C, prev_masks, unit_group, U, track, p, idx, count, status);
    if (s != RS3_OK) return s;
    return select_launch(z, dtype, G, m, n, C, prev_masks, unit_group, U, track, p, idx, count, nullptr, status, stream);
}

extern "C" rs3_status rs3_write_keepset(const uint8_t *seed_masks, const int32_t *unit_group, int U,
                                        int m, int n, const rs3_params *p, uint8_t *kw_out,
                                        int32_t *status, rs3_stream_t stream)
{
    if (!seed_masks || !unit_group || !p || !kw_out || !status) return RS3_EINVAL;
    if (U < 1 || m < 1 || n < 1 || p->D_w < 0) return RS3_EINVAL;
    if ((long)m * n > RS3_MAX_MN) return RS3_EUNSUPPORTED;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const size_t smem = 2 * (size_t)m * ((n + 31) / 32) * 4;
    if (rs3_kernel_smem((const void *)k_write_keepset, smem + 1024) != RS3_OK) return RS3_ECUDA;   // + its static arrays
    launch_pdl(k_write_keepset, dim3(U), dim3(SEL_THREADS), smem, st, seed_masks, unit_group, U, m, n, p->D_w,
               p->fall_lo, p->fall_hi, p->fall_through, p->union_mode, kw_out);
    if (cudaGetLastError() != cudaSuccess) return RS3_ECUDA;
    return RS3_OK;
}
