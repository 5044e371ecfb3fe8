// rs3_select.cu -- read-side keep-set K_r (Sec. 3.1: Eq. 1, 2, 4, 5) and the
// write keep-set K_w (Sec. 3.2: Eq. 8), integer-exact.
//
// k_select  the whole selection in one launch: a thread-block cluster of KC
//           CTAs per unit (per group in union mode).
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
//      kept cells in ascending order (block scan).
// Bound by latency and, in one CTA per SM, by instruction issue: 512 threads
// and no divisions in the loops, where 1024 threads took 30 000 cycles.
// One object of 64 x 64 cells and 256 channels takes 7.6 us in a graph, eight
// 14.0 us, and 16 streams x 3 objects of 96 x 96 20.9 us per call (7.3 us at the
// copy rate); 20.3, 25.9 and 59 us as three launches that passed the priors and
// the energies through global memory.
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

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// (.aligned: a warp's lanes execute it together, also after a loop or a branch
// that some of them left early)
__device__ __forceinline__ void cluster_arrive()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t dsmem_addr(const void *p, uint32_t rank)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void dsmem_st(uint32_t a, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t dsmem_ld(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

// A mask's cells as bit words: f(y, k, words k and k + 1 of row y), by every
// lane of the warp that loaded them (four rows of two words at a time).
template <typename F>
__device__ __forceinline__ void mask_words(const uint8_t *__restrict__ M, int m, int n, int WW, F f)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int yb = warp; yb < m; yb += 4 * SEL_WARPS)
        for (int k = 0; k < WW; k += 2) {
            const uint8_t *row = M + yb * n + 32 * k + lane;
            const bool in0 = 32 * k + lane < n, in1 = 32 * k + 32 + lane < n;
            uint8_t v0[4], v1[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const bool in = yb + q * SEL_WARPS < m;
                v0[q] = in && in0 ? __ldg(row + q * SEL_WARPS * n) : (uint8_t)0;
                v1[q] = in && in1 ? __ldg(row + q * SEL_WARPS * n + 32) : (uint8_t)0;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int y = yb + q * SEL_WARPS;
                if (y >= m) break;
                const uint32_t b0 = __ballot_sync(0xffffffffu, v0[q] != 0), b1 = __ballot_sync(0xffffffffu, v1[q] != 0);
                f(y, k, b0, b1);
            }
        }
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
    mask_words(M, m, n, WW, [&](int y, int k, uint32_t b0, uint32_t b1) {
        if (lane == 0) {
            a[y * WW + k] = b0;
            if (k + 1 < WW) a[y * WW + k + 1] = b1;
        }
        if (b0 | b1) {
            y0 = min(y0, y);
            y1 = max(y1, y);
            x0 = min(x0, 32 * k + (b0 ? __ffs(b0) - 1 : __ffs(b1) + 31));
            x1 = max(x1, 32 * k + (b1 ? 63 - __clz(b1) : 31 - __clz(b0)));
        }
    });
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
                if (remote) dsmem_st(key0 + 4 * j, __float_as_uint(r));
                else keys[j] = __float_as_uint(r);
            }
        }
    }
};

template <typename T>
__global__ void __launch_bounds__(SEL_THREADS)
k_select(const T *__restrict__ z, const uint8_t *__restrict__ masks, int m, int n, int C, int lpr,
         const int32_t *__restrict__ unit_group, int G, int U, rs3_track *__restrict__ track, int r_s, int c,
         int bbox_mode, int union_mode, int k, int KC, int32_t *__restrict__ idx, int32_t *__restrict__ count,
         int32_t *status)
{
    pdl_wait();
    extern __shared__ __align__(16) uint8_t sel_raw[];
    __shared__ uint32_t s_bin, s_rem, s_cnt, s_ncand, s_cand[32], s_mm[2][SEL_WARPS];
    const SelSmem S = sel_smem(m, n);
    uint32_t *P = reinterpret_cast<uint32_t *>(sel_raw + S.prior), *hist = P;
    uint32_t *A = reinterpret_cast<uint32_t *>(sel_raw + S.a), *keys = A;
    uint32_t *B = reinterpret_cast<uint32_t *>(sel_raw + S.b), *pref = B;
    uint16_t *list = reinterpret_cast<uint16_t *>(sel_raw + S.list);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int u = blockIdx.x / KC;
    const uint32_t rank = KC > 1 ? cluster_rank() : 0u;
    const int mn = m * n, WW = (n + 31) >> 5, words = m * WW;
    const int g = unit_group[u];
    if (g < 0 || g >= G) {                               // uniform over the cluster
        if (rank == 0 && threadIdx.x == 0) {
            latch_status(status, RS3_EINVAL);
            count[u] = 0;
        }
        return;
    }
    if (union_mode) {                                    // the group's first unit works for all of them
        bool other = false;
        for (int v = threadIdx.x; v < u; v += SEL_THREADS) other |= unit_group[v] == g;
        if (__syncthreads_or(other)) return;             // uniform over the cluster
    }
    const WordWalk walk(WW);
    for (int w = threadIdx.x; w < words; w += SEL_THREADS) P[w] = 0u;
    if (threadIdx.x == 0) s_ncand = 0u;
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
                for (int q = 0; q < KC; ++q) o |= dsmem_ld(dsmem_addr(P + w, (uint32_t)q));
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
    for (int y = warp; y < m; y += SEL_WARPS)
        for (int k = 0; k < WW; ++k) {
            const uint32_t bits = P[y * WW + k];
            if (bits >> lane & 1u) list[pref[y * WW + k] + __popc(bits & below)] = (uint16_t)(y * n + 32 * k + lane);
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
        if (lpr == 32) {
            constexpr int UN = sizeof(T) == 2 ? 8 : 4;
            for (uint32_t j0 = lo; j0 < hi; j0 += UN * SEL_WARPS) {
                Energies<T, UN> e;
                e.load(zg, list, j0, hi, C);
                if (!waited) {
                    cluster_wait();
                    waited = true;
                }
                e.store(keys, key0, KC > 1, j0, hi);
            }
        } else {
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
                if (!waited) {
                    cluster_wait();
                    waited = true;
                }
#pragma unroll
                for (int q = 0; q < UN; ++q) {
                    const uint32_t j = j0 + (q * SEL_WARPS + warp) * rpw + sub;
                    if (j < hi && l == 0) {
                        if (KC > 1) dsmem_st(key0 + 4 * j, __float_as_uint(s[q]));
                        else keys[j] = __float_as_uint(s[q]);
                    }
                }
            }
        }
        if (!waited) cluster_wait();
        if (KC > 1) {
            cluster_arrive();
            cluster_wait();
        }
    } else if (KC > 1) {
        cluster_wait();
    }
    if (rank != 0) return;
    if (!union_mode && threadIdx.x == 0) track[u] = tr;

    // keep key >= from, and the first `want` of key == equal
    uint32_t from = 0u, equal = 0xffffffffu, want = 0u;
    if (!keep_all && k > 0) {
        for (int b = threadIdx.x; b < SEL_BINS; b += SEL_THREADS) hist[b] = 0;
        __syncthreads();                                 // (KC = 1: the keys too)
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
        want = (uint32_t)k;
        int shift = max(0, 32 - __clz(span | 1u) - 11);
        for (;;) {
            for (uint32_t j = threadIdx.x; j < nP; j += SEL_THREADS) {
                const uint32_t d = keys[j] - base;       // wraps past every span for keys below base
                if (d <= span) atomicAdd(&hist[d >> shift], 1u);
            }
            __syncthreads();
            // thread t takes four bins, from the top
            const uint4 h = reinterpret_cast<const uint4 *>(hist)[SEL_BINS / 4 - 1 - threadIdx.x];
            uint32_t tot, above = block_excl_scan((h.x + h.y) + (h.z + h.w), tot);
            if (above < want && want <= above + (h.x + h.y) + (h.z + h.w)) {
                const uint32_t x[4] = {h.w, h.z, h.y, h.x};
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    if (above < want && want <= above + x[b]) {
                        s_bin = SEL_BINS - 1 - 4 * threadIdx.x - b;
                        s_rem = want - above;
                        s_cnt = x[b];
                    }
                    above += x[b];
                }
            }
            __syncthreads();
            base += s_bin << shift;
            want = s_rem;
            span = (1u << shift) - 1u;
            if (s_cnt == want) {                         // the whole bin is kept
                from = base;
                want = 0u;
                break;
            }
            if (shift == 0) {                            // a bin of equal keys
                from = base + 1u;
                equal = base;
                break;
            }
            if (s_cnt <= 32u) {                          // a warp ranks them (each for itself)
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
                const int at = __ffs(__ballot_sync(0xffffffffu, lane < nc && gt < want && want <= ge)) - 1;
                equal = __shfl_sync(0xffffffffu, x, at);
                from = equal + 1u;
                want -= __shfl_sync(0xffffffffu, gt, at);
                break;
            }
            shift = max(0, shift - 11);
            for (int b = threadIdx.x; b < SEL_BINS; b += SEL_THREADS) hist[b] = 0;
            __syncthreads();
        }
    }
    // each thread a run of the list; a kept cell's place is the number of kept
    // larger keys before it and of equal ones, of which the first `want` are kept
    const uint32_t per = (nP + SEL_THREADS - 1) / SEL_THREADS, j0 = threadIdx.x * per, j1 = min(j0 + per, nP);
    const bool ranked = !keep_all && k > 0;
    uint32_t off = j0;
    if (ranked) {
        uint32_t mine = 0, tot;
        for (uint32_t j = j0; j < j1; ++j) mine += (keys[j] >= from ? 0x10000u : 0u) + (keys[j] == equal ? 1u : 0u);
        off = block_excl_scan(mine, tot);
    }
    const auto emit = [&](int v) {
        int32_t *out = idx + (size_t)v * k;
        if (!ranked) {
            for (uint32_t j = threadIdx.x; j < n_kept; j += SEL_THREADS) out[j] = list[j];
        } else {
            uint32_t gt = off >> 16, eq = off & 0xffffu;
            for (uint32_t j = j0; j < j1; ++j) {
                const uint32_t key = keys[j];
                const bool is_eq = key == equal;
                if (key >= from || (is_eq && eq < want)) out[gt + min(eq, want)] = list[j];
                gt += key >= from ? 1u : 0u;
                eq += is_eq ? 1u : 0u;
            }
        }
        if (threadIdx.x == 0) count[v] = (int32_t)n_kept;
    };
    if (!union_mode) {
        emit(u);
    } else {
        for (int v0 = u; v0 < U; v0 += 32) {
            uint32_t in = __ballot_sync(0xffffffffu, v0 + lane < U && unit_group[min(v0 + lane, U - 1)] == g);
            for (; in; in &= in - 1) emit(v0 + __ffs(in) - 1);
        }
    }
}

// ---------------------------------------------------------------------------
// k_write_keepset: Eq. 8 with the 5% / 95% fall-through of Sec. 3.2, a CTA per
// unit on bit words: 64 x 64 cells, radius 12, took 16.5 us (cold) cell by cell.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(SEL_THREADS)
k_write_keepset(const uint8_t *__restrict__ seeds, const int32_t *__restrict__ unit_group, int U, int m, int n,
                int D_w, double fall_lo, double fall_hi, int fall_through, int union_mode, uint8_t *__restrict__ kw)
{
    pdl_wait();
    extern __shared__ __align__(16) uint8_t sel_raw[];
    const int mn = m * n, WW = (n + 31) >> 5, words = m * WW, u = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *a = reinterpret_cast<uint32_t *>(sel_raw), *b = a + words;
    const WordWalk walk(WW);
    mask_words(seeds + (size_t)u * mn, m, n, WW, [&](int y, int k, uint32_t b0, uint32_t b1) {
        if (lane == 0) {
            a[y * WW + k] = b0;
            if (k + 1 < WW) a[y * WW + k + 1] = b1;
        }
    });
    if (union_mode) {
        const int g = unit_group[u];
        for (int v0 = 0; v0 < U; v0 += 32) {
            uint32_t in = __ballot_sync(0xffffffffu, v0 + lane < U && v0 + lane != u && unit_group[min(v0 + lane, U - 1)] == g);
            for (; in; in &= in - 1)                       // (a word is always the same warp's)
                mask_words(seeds + (size_t)(v0 + __ffs(in) - 1) * mn, m, n, WW, [&](int y, int k, uint32_t b0, uint32_t b1) {
                    if (lane == 0) {
                        a[y * WW + k] |= b0;
                        if (k + 1 < WW) a[y * WW + k + 1] |= b1;
                    }
                });
        }
    }
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
    for (int y = warp; y < m; y += SEL_WARPS)
        for (int k = 0; k < WW; ++k)
            if (32 * k + lane < n) out[y * n + 32 * k + lane] = (uint8_t)(to[y * WW + k] >> lane & 1u);
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
// The selection keeps everything in shared memory; the size is that of a group
// bitmap, the priors and the energies in global memory, which callers allocate
// and rs3_select_queries_noalloc's limit counts.
extern "C" size_t rs3_select_workspace_bytes(int G, int U, int m, int n)
{
    if (G < 1 || U < 1 || m < 1 || n < 1) return 0;
    const size_t mn = (size_t)m * n;
    size_t off = align_up((size_t)G * ((mn + 31) / 32) * 4, 256);
    off = align_up(off + (size_t)U * mn, 256);
    return align_up(off + (size_t)G * mn * 4, 256);
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

rs3_status select_launch(const void *z, rs3_dtype dtype, int G, int m, int n, int C, const uint8_t *prev_masks,
                         const int32_t *unit_group, int U, rs3_track *track, const rs3_params *p, int32_t *idx,
                         int32_t *count, int32_t *status, rs3_stream_t stream)
{
    const int64_t k = rs3_kmax(p->rho, (int64_t)m * n);
    if (k < 0) return RS3_EINVAL;
    // CTAs per cluster: as many as are resident at once (two per SM), up to the
    // portable 8; 48 units of 96 x 96 cells: 20.9 us with 6 each, 22.6 with 4
    const long clusters = p->union_mode ? (G < U ? G : U) : U;
    const int KC = (int)std::min(8l, std::max(1l, 2l * rs3_sm_count() / clusters));
    const int nchunk = C / 8;
    const int lpr = nchunk >= 32 ? 32 : next_pow2(nchunk);
    const size_t smem = sel_smem(m, n).total;
    const void *fn = dtype == RS3_BF16 ? (const void *)k_select<uint16_t> : (const void *)k_select<float>;
    if (rs3_kernel_smem(fn, smem + 1024) != RS3_OK) return RS3_ECUDA;       // + the kernel's static arrays
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(U * KC));
    cfg.blockDim = dim3(SEL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = reinterpret_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = KC;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t e;
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
    return select_launch(z, dtype, G, m, n, C, prev_masks, unit_group, U, track, p, idx, count, status, stream);
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
    return select_launch(z, dtype, G, m, n, C, prev_masks, unit_group, U, track, p, idx, count, status, stream);
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
