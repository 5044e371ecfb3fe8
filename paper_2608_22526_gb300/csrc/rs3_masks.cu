// rs3_masks.cu -- the decoder side and the pixel-space front end of RS3-Prune.
//
//   rs3_close_argmax     Sec. 3.3: per-object closure of the decoder's binary
//                        masks with a (2R+1)^2 square (9 x 9 in the paper),
//                        then the per-pixel argmax over a stream's objects
//                        (the palette mask); optionally down_s of each closed
//                        mask onto the token grid (Sec. 3.1, Eq. 2's input)
//   rs3_seed_from_masks  Sec. 3.1, Eq. 1: the seed box of each object's pixel
//                        mask projected onto the grid (the tracker state of
//                        Eq. 4), with down_s of the mask and the filled box
//
// Closure.  A CTA of 16 warps owns a tile of up to 24 rows x NS strips of 128
// columns of one stream's decoder output (NS = 1..4, the whole width up to 512
// columns) and takes the stream's objects one after the other.  A warp reads a
// row of a strip with one 16-byte load per lane, so its four ballots (logit >
// 0) hold the strip's bits by column modulo 4: bit l of word c is column 4 l +
// c.  In that layout a horizontal shift by d = 4 q + b columns is a shift by q
// bits of another word, and for the paper's radius of 4 a dilation is two
// funnel shifts per word of running ORs.  The tile plus a halo of 2R rows above
// and below and a strip on each side is thresholded into shared memory, then
// four separable passes (horizontal and vertical dilation, horizontal and
// vertical erosion) run on 128 columns per thread and step.  The object is a
// set of the unbounded plane with nothing set outside the image: pixels outside
// are zero bits, and the dilation is evaluated there too, so the erosion never
// treats the border as set or unset by convention.  With R <= 8 every bit the
// tile's result depends on lies within 2R = 16 pixels of the tile.  Per pixel
// the largest logit among the objects whose closed mask holds it stays in
// shared memory (equal logits keep the earlier object).
//
// Where a stream has few tiles, a thread-block cluster of KC <= 8 CTAs shares
// one: rank r closes objects r, r + KC, ..., and each rank merges a share of
// the tile's rows from all ranks' shared memory (DSMEM), equal logits going to
// the object listed first.  close_shape() picks rows and KC.
//
// Each logit is read from DRAM once; halo re-reads by neighbouring tiles hit
// L2.  16 streams x 3 objects of 384 x 384 (31 MB, 4.6 us at the copy rate): 19.1
// us per call, half of the issue slots busy, mostly with the thresholds, the
// argmax and its labels (at two CTAs per SM three strips spill 120 bytes per
// thread, four 40); 91 us with a scalar load and a ballot per 32 pixels,
// general funnel-shift dilations and an 8-row halo per 16 rows on CTAs that
// filled 1.3 waves.  8 objects of 1024 x 1024: 79 -> 29 us.
#include "rs3_cluster.cuh"
#include "rs3_internal.cuh"

#include <algorithm>
#include <atomic>
#include <climits>
#include <mutex>

namespace {

constexpr int CA_WARPS = 16;
constexpr int CA_THREADS = 32 * CA_WARPS;
constexpr int CA_RMAX = 8;
constexpr int CA_ROWS = 24;         // the most rows of a tile
constexpr int CA_KCMAX = 8;         // CTAs of a cluster (the portable size)

// word e of a strip shifted so that bit l holds column 4 (l + q) + e; pv and
// nx are the same word of the strips to the left and right
__device__ __forceinline__ uint32_t strip_shift(uint32_t pv, uint32_t x, uint32_t nx, int q)
{
    return q == 0 ? x : q > 0 ? __funnelshift_r(x, nx, q) : __funnelshift_l(pv, x, -q);
}

// Bits ORed (DIL) or ANDed over horizontal shifts -R..R of one strip with its
// neighbours.  RC = 4: columns 4 l + c - 4 .. 4 l + c + 4 are words c..3 of
// lane l - 1, every word of lane l and words 0..c of lane l + 1, so running
// ORs (ANDs) from either end and one shift each way do.  RC = 0 takes any
// radius up to 8 from R.
template <bool DIL>
__device__ __forceinline__ uint32_t comb(uint32_t a, uint32_t b) { return DIL ? (a | b) : (a & b); }

template <bool DIL, int RC>
__device__ __forceinline__ uint4 horizontal(uint4 pv, uint4 x, uint4 nx, int R)
{
    const uint32_t p[4] = {pv.x, pv.y, pv.z, pv.w}, o[4] = {x.x, x.y, x.z, x.w}, n[4] = {nx.x, nx.y, nx.z, nx.w};
    uint32_t r[4];
    if (RC == 4) {
        uint32_t lo[4], lon[4], hi[4], hip[4];       // words 0..c and c..3
        lo[0] = o[0]; lon[0] = n[0]; hi[3] = o[3]; hip[3] = p[3];
#pragma unroll
        for (int c = 1; c < 4; ++c) {
            lo[c] = comb<DIL>(lo[c - 1], o[c]);
            lon[c] = comb<DIL>(lon[c - 1], n[c]);
            hi[3 - c] = comb<DIL>(hi[4 - c], o[3 - c]);
            hip[3 - c] = comb<DIL>(hip[4 - c], p[3 - c]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
            r[c] = comb<DIL>(lo[3], comb<DIL>(__funnelshift_l(hip[c], hi[c], 1), __funnelshift_r(lo[c], lon[c], 1)));
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) r[c] = o[c];
#pragma unroll
        for (int q = -2; q <= 2; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t w = strip_shift(p[e], o[e], n[e], q);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int d = 4 * q + e - c;
                    if ((d < 0 ? -d : d) <= R) r[c] = comb<DIL>(r[c], w);
                }
            }
    }
    return make_uint4(r[0], r[1], r[2], r[3]);
}

template <bool DIL>
__device__ __forceinline__ uint4 comb4(uint4 a, uint4 b)
{
    return make_uint4(comb<DIL>(a.x, b.x), comb<DIL>(a.y, b.y), comb<DIL>(a.z, b.z), comb<DIL>(a.w, b.w));
}

// four adjacent logits of a row; VEC: the logits start on a 16-byte boundary
// (every row then does: w is a multiple of 32)
template <bool VEC>
__device__ __forceinline__ float4 load_logits(const float *p)
{
    if (VEC) return __ldg(reinterpret_cast<const float4 *>(p));
    return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}

// four adjacent bytes; VEC: the array starts on a 4-byte boundary
template <bool VEC>
__device__ __forceinline__ void store_bytes(uint8_t *p, uint32_t v)
{
    if (VEC) {
        *reinterpret_cast<uint32_t *>(p) = v;
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) p[c] = (uint8_t)(v >> 8 * c);
    }
}

// a strip's row -> its four words (lane 0 stores)
__device__ __forceinline__ void store_bits(uint4 *dst, float4 v, int lane)
{
    const uint32_t b0 = __ballot_sync(0xffffffffu, v.x > 0.f), b1 = __ballot_sync(0xffffffffu, v.y > 0.f);
    const uint32_t b2 = __ballot_sync(0xffffffffu, v.z > 0.f), b3 = __ballot_sync(0xffffffffu, v.w > 0.f);
    if (lane == 0) *dst = make_uint4(b0, b1, b2, b3);
}

// Shared memory of a CTA, in 16-byte words: bits of window rows x (NS + 2)
// strips (thresholded, dilated along rows, dilated), of the erosion along rows,
// the closure; the best logits and labels (a byte each, 0 = none) per pixel.
template <int NS, int RM>
struct CloseSmem {
    static constexpr int NR = CA_ROWS + 4 * RM, SW = NS + 2;
    static constexpr int A = 0, H = A + NR * SW, D = H + NR * SW, E = D + NR * SW;
    static constexpr int C = E + (CA_ROWS + 2 * RM) * NS;
    static constexpr int BV = C + CA_ROWS * NS;                    // float4 [rows NS][32]
    static constexpr int BL = BV + CA_ROWS * NS * 32;              // uint32 [rows NS][32]
    static constexpr int BYTES = 16 * (BL + CA_ROWS * NS * 8);
};

// One tile of `rows` rows x NS strips.  KC > 1: the CTAs of a cluster share the
// stream's objects.  RC = 4 fixes the radius at compile time (the paper's 9 x 9
// element), RC = 0 takes it from R_rt.  VEC: aligned arrays.
template <int NS, int RC, bool VEC>
__global__ void __launch_bounds__(CA_THREADS, RC > 0 ? 2 : 1)
k_close_argmax(const float *__restrict__ logits, const int32_t *__restrict__ gstart, int U, int h,
               int w, int R_rt, int s, int rows, int KC, uint8_t *__restrict__ palette, uint8_t *__restrict__ closed,
               uint8_t *__restrict__ grid, int32_t *status)
{
    const int R = RC > 0 ? RC : R_rt;
    constexpr int RM = RC > 0 ? RC : CA_RMAX;
    using M = CloseSmem<NS, RM>;
    constexpr int SW = M::SW;                              // window strips [s0 - 1, s0 + NS + 1)
    constexpr int NT = (CA_ROWS * NS + CA_WARPS - 1) / CA_WARPS;   // tile rows x strips of a warp, at most
    constexpr int NH = (4 * RM * NS + CA_WARPS - 1) / CA_WARPS;    // halo rows x strips of a warp
    extern __shared__ uint4 ca_smem[];
    uint4 *sA = ca_smem + M::A, *sH = ca_smem + M::H, *sD = ca_smem + M::D, *sE = ca_smem + M::E, *sC = ca_smem + M::C;
    float4 *sBV = reinterpret_cast<float4 *>(ca_smem + M::BV);
    uint32_t *sBL = reinterpret_cast<uint32_t *>(ca_smem + M::BL);
    pdl_wait();
    const uint32_t rank = KC > 1 ? cluster_rank() : 0u;
    const int g = blockIdx.z / KC;
    const int r0 = blockIdx.y * rows, x0 = blockIdx.x * NS * 128;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int u0 = gstart[g], u1 = gstart[g + 1];
    // the same values reach every CTA of the cluster, so all of them leave
    // here together, before any cluster barrier
    if (u0 < 0 || u1 < u0 || u1 > U || u1 - u0 > 255) {
        if (t == 0 && rank == 0) latch_status(status, RS3_EINVAL);
        return;
    }
    const int brv = min(rows, h - r0);                     // tile rows inside the image
    const int nwin = rows + 4 * R;                         // window rows [r0 - 2R, r0 + rows + 2R)
    const bool sides = x0 > 0 || x0 + NS * 128 < w;        // columns beside the tile lie in the image
    if (!sides)
        for (int p = t; p < 2 * nwin; p += CA_THREADS) sA[(p >> 1) * SW + (p & 1) * (NS + 1)] = make_uint4(0u, 0u, 0u, 0u);
    // where this lane's pixels lie in an object's image (-1: outside): the
    // tile's rows, and the halo rows (the first 2R above the tile, the rest below)
    int off[NT], hoff[NH], goff[NT];
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int p = warp + CA_WARPS * i, x = x0 + (p % NS) * 128 + 4 * lane;
        off[i] = p < brv * NS && x < w ? (r0 + p / NS) * w + x : -1;
        goff[i] = -1;
    }
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        const int p = warp + CA_WARPS * i, j = p / NS, x = x0 + (p % NS) * 128 + 4 * lane;
        const int row = r0 - 2 * R + (j < 2 * R ? j : rows + j);
        hoff[i] = j < 4 * R && row >= 0 && row < h && x < w ? row * w + x : -1;
    }
    int gm = 0, gn = 0;
    // for s >= 4 their grid cell (4 cell + which of the four columns it takes);
    // its divisions run while the first object's logits are on their way
    const auto grid_cells = [&]() {
        gm = h / s;
        gn = w / s;
        const int gi0 = (r0 + s - 1) / s;                  // first grid row of the tile
        uint32_t grows = 0u;                               // which of its rows are grid rows
        if (grid && s >= 4)
            for (int k = gi0 * s - r0; k < brv; k += s) grows |= 1u << k;
        constexpr int NX = NS == 3 ? 3 : 1;                // a warp's tasks lie in one strip, unless NS = 3
        int gx4[NX];
#pragma unroll
        for (int k = 0; k < NX; ++k) {
            const int x = x0 + (NX == 1 ? warp % NS : k) * 128 + 4 * lane, gx = (x + s - 1) / s, c = gx * s - x;
            gx4[k] = c < 4 ? 4 * gx + c : -1;
        }
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            const int p = warp + CA_WARPS * i, k = p / NS;
            const int gx = NX == 1 ? gx4[0] : p % NS == 0 ? gx4[0] : p % NS == 1 ? gx4[1 % NX] : gx4[2 % NX];
            goff[i] = off[i] >= 0 && gx >= 0 && (grows >> k & 1u) ? 4 * (gi0 + __popc(grows & ((1u << k) - 1u))) * gn + gx : -1;
        }
    };
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t lane_bit = 1u << lane;
    for (int u = u0 + (int)rank; u < u1; u += KC) {
        const float *L = logits + (size_t)u * h * w;
        // 1. all of the object's loads, then its ballots: the tile, the halo
        //    and, in images wider than the tile, the 16 columns on either side
        float4 v[NT], hv[NH];
#pragma unroll
        for (int i = 0; i < NT; ++i) v[i] = off[i] >= 0 ? load_logits<VEC>(L + off[i]) : none;
#pragma unroll
        for (int i = 0; i < NH; ++i) hv[i] = hoff[i] >= 0 ? load_logits<VEC>(L + hoff[i]) : none;
        if (u == u0 + (int)rank) grid_cells();
        uint8_t *gu = grid + (size_t)u * gm * gn;
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            const int p = warp + CA_WARPS * i;
            if (p < rows * NS) store_bits(&sA[(2 * R + p / NS) * SW + 1 + p % NS], v[i], lane);
        }
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const int p = warp + CA_WARPS * i, j = p / NS;
            if (j < 4 * R) store_bits(&sA[(j < 2 * R ? j : rows + j) * SW + 1 + p % NS], hv[i], lane);
        }
        if (sides) {
            // lanes 28..31 read the strip to the left, lanes 0..3 the one to the right
            for (int lr = warp; lr < nwin; lr += CA_WARPS) {
                const int row = r0 - 2 * R + lr, x = lane >= 28 ? x0 - 128 + 4 * lane : x0 + NS * 128 + 4 * lane;
                const bool in = (lane < 4 || lane >= 28) && row >= 0 && row < h && x >= 0 && x < w;
                const float4 sv = in ? load_logits<VEC>(L + (size_t)row * w + x) : none;
                const uint32_t b0 = __ballot_sync(0xffffffffu, sv.x > 0.f), b1 = __ballot_sync(0xffffffffu, sv.y > 0.f);
                const uint32_t b2 = __ballot_sync(0xffffffffu, sv.z > 0.f), b3 = __ballot_sync(0xffffffffu, sv.w > 0.f);
                if (lane < 2) {
                    const uint32_t k = lane ? 0xfu : 0xf0000000u;
                    sA[lr * SW + lane * (NS + 1)] = make_uint4(b0 & k, b1 & k, b2 & k, b3 & k);
                }
            }
        }
        __syncthreads();
        // 2. horizontal dilation on every window strip (the outermost strips'
        //    missing neighbours are read as zero: only their bits next to the
        //    tile are used below, and those do not depend on them)
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        for (int p = t; p < nwin * SW; p += CA_THREADS) {
            const int ls = p % SW;
            sH[p] = horizontal<true, RC>(ls > 0 ? sA[p - 1] : zero, sA[p], ls < SW - 1 ? sA[p + 1] : zero, R);
        }
        __syncthreads();
        // 3. vertical dilation, window rows [R, rows + 3R)
        for (int p = R * SW + t; p < (rows + 3 * R) * SW; p += CA_THREADS) {
            uint4 r = sH[p];
#pragma unroll
            for (int d = 1; d <= R; ++d) r = comb4<true>(r, comb4<true>(sH[p - d * SW], sH[p + d * SW]));
            sD[p] = r;
        }
        __syncthreads();
        // 4. horizontal erosion of the tile's strips, window rows [R, rows + 3R)
        for (int p = t; p < (rows + 2 * R) * NS; p += CA_THREADS) {
            const uint4 *d = sD + (R + p / NS) * SW + p % NS;
            sE[p] = horizontal<false, RC>(d[0], d[1], d[2], R);
        }
        __syncthreads();
        // 5. vertical erosion: the closure of the tile's rows
        for (int p = t; p < rows * NS; p += CA_THREADS) {
            uint4 r = sE[p + R * NS];
#pragma unroll
            for (int d = 1; d <= R; ++d) r = comb4<false>(r, comb4<false>(sE[p + (R - d) * NS], sE[p + (R + d) * NS]));
            sC[p] = r;
        }
        __syncthreads();
        // 6. argmax update, closed mask and its down_s onto the grid
        const uint32_t lab = (uint32_t)(u - u0 + 1);
        const bool first = u == u0 + (int)rank;
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            const int p = warp + CA_WARPS * i;
            if (p >= rows * NS) continue;
            const uint4 cw = sC[p];
            const bool bit[4] = {(cw.x & lane_bit) != 0, (cw.y & lane_bit) != 0, (cw.z & lane_bit) != 0,
                                 (cw.w & lane_bit) != 0};
            const uint32_t bytes = (uint32_t)bit[0] | (uint32_t)bit[1] << 8 | (uint32_t)bit[2] << 16 | (uint32_t)bit[3] << 24;
            // a pixel without a label takes the object's whatever its logit
            if (first) {
                sBV[p * 32 + lane] = v[i];
                sBL[p * 32 + lane] = bytes * lab;
            } else if ((cw.x | cw.y | cw.z | cw.w) != 0u) {    // (the same for the warp)
                const float vv[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
                const float4 best = sBV[p * 32 + lane];
                float bv[4] = {best.x, best.y, best.z, best.w};
                uint32_t bl = sBL[p * 32 + lane];
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (bit[c] && (vv[c] > bv[c] || (bl & 255u << 8 * c) == 0u)) {
                        bv[c] = vv[c];
                        bl = __byte_perm(bl, lab, c == 0 ? 0x3214 : c == 1 ? 0x3240 : c == 2 ? 0x3410 : 0x4210);
                    }
                sBV[p * 32 + lane] = make_float4(bv[0], bv[1], bv[2], bv[3]);
                sBL[p * 32 + lane] = bl;
            }
            if (closed && off[i] >= 0) store_bytes<VEC>(closed + (size_t)u * h * w + off[i], bytes);
            if (goff[i] >= 0) gu[goff[i] >> 2] = (uint8_t)(bytes >> 8 * (goff[i] & 3) & 1u);
            if (grid && s < 4 && off[i] >= 0) {            // several cells in the lane's four columns
                const int row = r0 + p / NS, x = x0 + (p % NS) * 128 + 4 * lane;
                const auto over_s = [s](int a) { return s == 1 ? a : s == 2 ? a >> 1 : a / 3; };
                const int gy = over_s(row);
                if (gy * s == row)
                    for (int gx = over_s(x + s - 1); gx * s < x + 4; ++gx)
                        gu[gy * gn + gx] = (uint8_t)(bytes >> 8 * (gx * s - x) & 1u);
            }
        }
    }
    if (u0 + (int)rank >= u1)                              // no object: nothing written above
        for (int p = warp; p < rows * NS; p += CA_WARPS) sBL[p * 32 + lane] = 0u;
    if (KC > 1) {
        // 7. rank r merges rows (of a strip) r, r + KC, ... of the tile: the
        //    larger logit, the lower label on equal logits (each rank's best
        //    already holds its lowest label among equal logits)
        cluster_barrier();
        for (int p = warp * KC + (int)rank; p < rows * NS; p += CA_WARPS * KC) {
            float b[4] = {0.f, 0.f, 0.f, 0.f};
            uint32_t bl = 0u;
            float4 v2[8];
            uint32_t l2[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < KC) {
                    v2[q] = dsmem_ld_f32x4(dsmem_addr(sBV + p * 32 + lane, (uint32_t)q));
                    l2[q] = dsmem_ld_u32(dsmem_addr(sBL + p * 32 + lane, (uint32_t)q));
                }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < KC) {
                    const float vq[4] = {v2[q].x, v2[q].y, v2[q].z, v2[q].w};
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint32_t ln = l2[q] >> 8 * c & 255u, lo = bl >> 8 * c & 255u;
                        if (ln != 0u && (lo == 0u || vq[c] > b[c] || (vq[c] == b[c] && ln < lo))) {
                            b[c] = vq[c];
                            bl = (bl & ~(255u << 8 * c)) | ln << 8 * c;
                        }
                    }
                }
            const int row = r0 + p / NS, x = x0 + (p % NS) * 128 + 4 * lane;
            if (palette && row < h && x < w) store_bytes<VEC>(palette + ((size_t)g * h + row) * w + x, bl);
        }
        cluster_barrier();       // no CTA leaves while another reads its shared memory
    } else if (palette) {
#pragma unroll
        for (int i = 0; i < NT; ++i)
            if (off[i] >= 0) store_bytes<VEC>(palette + (size_t)g * h * w + off[i], sBL[(warp + CA_WARPS * i) * 32 + lane]);
    }
}

// ---------------------------------------------------------------------------
// Seed box and down_s of pixel masks
// ---------------------------------------------------------------------------
// Masks of up to about 1 MB take one launch (k_seed): the KC <= 8 CTAs of a cluster
// share a unit's rows.  Each finds its band's extreme rows and columns, the boxes
// meet through DSMEM, then the first CTA writes the tracker and each its share of
// the grid mask and of the filled grid box.  Bound by latency (3 us of launch,
// barriers and reductions) and by what one SM can read, about 35 GB/s when all of
// a cluster's do: larger masks are spread over all SMs, in three launches.
constexpr int SEED_KC = 8, SEED_BATCH = 8;
constexpr int SCAN_THREADS = 256, SCAN_CHUNKS = SCAN_THREADS * SEED_BATCH;   // k_seed_scan: a CTA's chunks, about

// The extreme set rows and columns (y0, x0, y1, x1) of rows [r0, r0 + nr) of a mask
// of cpr 16-byte chunks per row, by a CTA; in every lane of its first warp.  `dx` is
// blockDim.x modulo cpr.  Eight loads in flight per thread; byte j of a chunk is
// column 16 c + j.  A thread's chunks ascend, so its first and last set ones give
// its rows, and only a chunk that reaches past the columns seen so far is looked into.
__device__ __forceinline__ int4 band_box(const uint8_t *__restrict__ M, int r0, int nr, uint32_t cpr, uint32_t dx)
{
    __shared__ int4 s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint4 *base = reinterpret_cast<const uint4 *>(M + (size_t)r0 * cpr * 16);
    const uint32_t chunks = (uint32_t)nr * cpr, T = blockDim.x;
    uint32_t first = 0xffffffffu, last = 0u;                 // set chunks
    int x0 = INT_MAX, x1 = -1;
    uint32_t cx = threadIdx.x % cpr;                         // the next chunk's column
    for (uint32_t c0 = threadIdx.x; c0 < chunks; c0 += SEED_BATCH * T) {
        uint4 v[SEED_BATCH];
#pragma unroll
        for (int k = 0; k < SEED_BATCH; ++k)
            v[k] = c0 + k * T < chunks ? __ldg(base + c0 + k * T) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int k = 0; k < SEED_BATCH; ++k) {
            if ((v[k].x | v[k].y | v[k].z | v[k].w) != 0u) {
                last = c0 + k * T;
                first = min(first, last);
                const int xb = 16 * (int)cx;
                if (xb < x0 || xb + 15 > x1) {
                    const uint32_t wd[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t nz = __vcmpne4(wd[j], 0u);     // 0xff in every non-zero byte
                        if (nz) {
                            x0 = min(x0, xb + 4 * j + ((__ffs(nz) - 1) >> 3));
                            x1 = max(x1, xb + 4 * j + ((31 - __clz(nz)) >> 3));
                        }
                    }
                }
            }
            cx += dx;
            if (cx >= cpr) cx -= cpr;
        }
    }
    int y0 = INT_MAX, y1 = -1;
    if (x1 >= 0) {
        y0 = r0 + (int)(first / cpr);
        y1 = r0 + (int)(last / cpr);
    }
    y0 = __reduce_min_sync(0xffffffffu, y0);
    x0 = __reduce_min_sync(0xffffffffu, x0);
    y1 = __reduce_max_sync(0xffffffffu, y1);
    x1 = __reduce_max_sync(0xffffffffu, x1);
    if (lane == 0) s_warp[warp] = make_int4(y0, x0, y1, x1);
    __syncthreads();
    int4 b = s_warp[lane < nw ? lane : 0];
    if (warp == 0)
        b = make_int4(__reduce_min_sync(0xffffffffu, b.x), __reduce_min_sync(0xffffffffu, b.y),
                      __reduce_max_sync(0xffffffffu, b.z), __reduce_max_sync(0xffffffffu, b.w));
    return b;
}

// Sizes of a call that the kernels would divide for.
struct SeedDims {
    int h, w, s, m, n;
    int rows;            // image rows per CTA
    uint32_t cpr, dx;    // chunks per row; threads of a CTA modulo that
    uint32_t share;      // grid cells per CTA
};

__device__ __forceinline__ uint8_t in_box(const rs3_track &t, uint32_t c, int n)
{
    const int i = (int)(c / (uint32_t)n), j = (int)(c - (uint32_t)i * n);
    return t.valid && i >= t.y0 && i <= t.y1 && j >= t.x0 && j <= t.x1;
}

__global__ void __launch_bounds__(512)
k_seed(const uint8_t *__restrict__ masks, SeedDims d, int KC, rs3_track *__restrict__ track, uint8_t *__restrict__ grid,
       uint8_t *__restrict__ box)
{
    pdl_wait();
    __shared__ int4 s_box;                                   // (y0, x0, y1, x1)
    const int u = blockIdx.y, lane = threadIdx.x & 31;
    const uint32_t rank = KC > 1 ? cluster_rank() : 0u, T = blockDim.x;
    const uint8_t *M = masks + (size_t)u * d.h * d.w;
    const int r0 = min((int)rank * d.rows, d.h), nr = min(d.rows, d.h - r0);
    const int4 b = band_box(M, r0, nr, d.cpr, d.dx);
    if (threadIdx.x == 0) s_box = b;
    if (KC > 1) cluster_arrive();                            // (orders s_box within the CTA too)
    else __syncthreads();
    // beside the other CTAs' arrivals
    const uint32_t cells = (uint32_t)d.m * d.n, ca = min(rank * d.share, cells), cb = min(ca + d.share, cells);
    if (grid)
        for (uint32_t c = ca + threadIdx.x; c < cb; c += T) {
            const uint32_t i = c / (uint32_t)d.n, j = c - i * d.n;
            grid[(size_t)u * cells + c] = M[(size_t)i * d.s * d.w + (size_t)j * d.s] != 0;
        }
    int y0, x0, y1, x1;
    if (KC > 1) {
        cluster_wait();
        const uint32_t from = dsmem_addr(&s_box, lane < KC ? lane : 0u);
        y0 = __reduce_min_sync(0xffffffffu, (int)dsmem_ld_u32(from));
        x0 = __reduce_min_sync(0xffffffffu, (int)dsmem_ld_u32(from + 4u));
        y1 = __reduce_max_sync(0xffffffffu, (int)dsmem_ld_u32(from + 8u));
        x1 = __reduce_max_sync(0xffffffffu, (int)dsmem_ld_u32(from + 12u));
        cluster_arrive();
    } else {
        y0 = s_box.x; x0 = s_box.y; y1 = s_box.z; x1 = s_box.w;
    }
    // the pixel box divided by s (rounding down); no pixels: all zeros
    rs3_track t = {0, 0, 0, 0, 0, 0};
    if (y1 >= 0) t = rs3_track{y0 / d.s, x0 / d.s, y1 / d.s, x1 / d.s, 1, 0};
    if (rank == 0 && threadIdx.x == 0) track[u] = t;
    if (box)
        for (uint32_t c = ca + threadIdx.x; c < cb; c += T) box[(size_t)u * cells + c] = in_box(t, c, d.n);
    if (KC > 1) cluster_wait();                              // no CTA leaves while another reads its box
}

// The three launches of larger masks.  The box is divided by s before it is merged
// (rounding down keeps the order), so the tracker is in its final state after the
// scan, but for the units without a set pixel.
__global__ void k_seed_init(rs3_track *track, int U)
{
    pdl_wait();
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u < U) track[u] = rs3_track{INT_MAX, INT_MAX, -1, -1, 0, 0};
}

// A CTA per band of rows and unit: its box, merged into the unit's tracker with
// atomics, and its rows of the grid mask.
__global__ void __launch_bounds__(SCAN_THREADS)
k_seed_scan(const uint8_t *__restrict__ masks, SeedDims d, rs3_track *track, uint8_t *__restrict__ grid)
{
    pdl_wait();
    const int u = blockIdx.y, r0 = blockIdx.x * d.rows, nr = min(d.rows, d.h - r0);
    const uint8_t *M = masks + (size_t)u * d.h * d.w;
    const int4 b = band_box(M, r0, nr, d.cpr, d.dx);
    if (threadIdx.x == 0 && b.z >= 0) {
        atomicMin(&track[u].y0, b.x / d.s);
        atomicMin(&track[u].x0, b.y / d.s);
        atomicMax(&track[u].y1, b.z / d.s);
        atomicMax(&track[u].x1, b.w / d.s);
        track[u].valid = 1;
    }
    if (!grid) return;
    const int i0 = (r0 + d.s - 1) / d.s, i1 = min((r0 + nr + d.s - 1) / d.s, d.m);
    for (uint32_t c = threadIdx.x; c < (uint32_t)(i1 - i0) * d.n; c += SCAN_THREADS) {
        const uint32_t i = c / (uint32_t)d.n, j = c - i * d.n;
        grid[((size_t)u * d.m + i0 + i) * d.n + j] = M[(size_t)(i0 + i) * d.s * d.w + (size_t)j * d.s] != 0;
    }
}

// The filled grid box, and zeros for the tracker of a unit without a set pixel
// (written by one thread: the others read `valid` alone of it, which stays 0).
__global__ void __launch_bounds__(SCAN_THREADS)
k_seed_finish(SeedDims d, rs3_track *track, uint8_t *__restrict__ box)
{
    pdl_wait();
    const int u = blockIdx.y;
    rs3_track t = {0, 0, 0, 0, 0, 0};
    if (track[u].valid) t = track[u];
    else if (blockIdx.x == 0 && threadIdx.x == 0) track[u] = t;
    const uint32_t cells = (uint32_t)d.m * d.n, c0 = blockIdx.x * d.share, c1 = min(c0 + d.share, cells);
    if (box)
        for (uint32_t c = c0 + threadIdx.x; c < c1; c += SCAN_THREADS) box[(size_t)u * cells + c] = in_box(t, c, d.n);
}

}  // namespace

struct CloseShape {
    int ns, rows, KC, tiles_x;
};

// Clusters of 1..8 CTAs of a kernel that are resident at once on the current
// device (fit[KC]); asked from the runtime at the kernel's first call there, which
// also raises its shared-memory limit.  A cluster lies within one GPC, so they are
// fewer than the CTAs that fit divided by KC: 36 of 8 CTAs where 304 CTAs fit.
template <int NS, int RC, bool VEC>
static const int *close_fit()
{
    constexpr int smem = CloseSmem<NS, (RC > 0 ? RC : CA_RMAX)>::BYTES;
    static std::mutex mu;
    static std::atomic<bool> ready[64];
    static int fit[64][CA_KCMAX + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (ready[dev].load(std::memory_order_acquire)) return fit[dev];
    std::lock_guard<std::mutex> lock(mu);
    const auto kernel = k_close_argmax<NS, RC, VEC>;
    if (rs3_kernel_smem((const void *)kernel, smem) != RS3_OK) return nullptr;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, CA_THREADS, smem) != cudaSuccess || per_sm < 1)
        return nullptr;
    fit[dev][1] = per_sm * rs3_sm_count();
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = attr.val.clusterDim.y = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(CA_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    for (int KC = 2; KC <= CA_KCMAX; ++KC) {
        attr.val.clusterDim.z = KC;
        cfg.gridDim = dim3(1, 1, KC);
        if (cudaOccupancyMaxActiveClusters(&fit[dev][KC], kernel, &cfg) != cudaSuccess) return nullptr;
    }
    ready[dev].store(true, std::memory_order_release);
    return fit[dev];
}

// Rows per tile and CTAs per cluster: the least waves x objects per CTA x cost
// of an object, where the cost counts the strip rows read (halo and all) and a
// fixed part for the passes' latency, worth about 40 of them.  fit[KC] clusters
// of KC CTAs are resident; the rows tried are those that just fill one wave (at
// least 6: fewer are no faster), 16 and 24, and the KC those that leave a CTA
// fewer objects.  8 objects of one stream at 256 x 256: 7.1 us in 8-row tiles of
// 32 clusters, 10.1 in 37 clusters of 7-row tiles, one more than are resident; at
// 1024 x 1024 28.8 and 42.1.
static CloseShape close_shape(int G, int objects, int h, int w, int R, const int *fit)
{
    CloseShape best = {};
    best.ns = std::min(4, (w + 127) / 128);
    best.tiles_x = (w + 128 * best.ns - 1) / (128 * best.ns);
    const long long columns = (long long)best.tiles_x * G;              // tiles per row of tiles
    double least = 0.0;
    for (int KC = 1; KC <= objects; ++KC) {
        const int per_cta = (objects + KC - 1) / KC;
        if (fit[KC] < 1 || (KC > 1 && per_cta == (objects + KC - 2) / (KC - 1))) continue;
        const int tiles = (int)std::max(1ll, fit[KC] / columns);
        const int one_wave = std::min(CA_ROWS, std::max(6, (h + tiles - 1) / tiles));
        for (const int rows : {one_wave, 16, CA_ROWS}) {
            const long long n = columns * ((h + rows - 1) / rows);
            const double cost = (double)((n + fit[KC] - 1) / fit[KC]) * per_cta *
                                    (40.0 + (double)(rows + 4 * R) * best.ns) + (KC > 1 ? 20.0 : 0.0);
            if (best.KC == 0 || cost < least) {
                least = cost;
                best.rows = rows;
                best.KC = KC;
            }
        }
    }
    return best;
}

template <int NS, int RC, bool VEC>
static cudaError_t launch_close(int G, int objects, int h, cudaStream_t st, const float *logits, const int32_t *gstart,
                                int U, int w, int R, int s, uint8_t *palette, uint8_t *closed, uint8_t *grid,
                                int32_t *status)
{
    const int *fit = close_fit<NS, RC, VEC>();
    if (!fit) return cudaErrorInvalidValue;
    const CloseShape c = close_shape(G, objects, h, w, R, fit);
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(CA_THREADS);
    cfg.dynamicSmemBytes = CloseSmem<NS, (RC > 0 ? RC : CA_RMAX)>::BYTES;
    cfg.gridDim = dim3(c.tiles_x, (h + c.rows - 1) / c.rows, G * c.KC);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = c.KC;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k_close_argmax<NS, RC, VEC>, logits, gstart, U, h, w, R, s, c.rows, c.KC, palette,
                              closed, grid, status);
}

template <int RC, bool VEC, typename... Args>
static cudaError_t launch_close_strips(int G, int objects, int h, cudaStream_t st, const float *logits,
                                       const int32_t *gstart, int U, int w, Args... args)
{
    switch (std::min(4, (w + 127) / 128)) {
    case 1: return launch_close<1, RC, VEC>(G, objects, h, st, logits, gstart, U, w, args...);
    case 2: return launch_close<2, RC, VEC>(G, objects, h, st, logits, gstart, U, w, args...);
    case 3: return launch_close<3, RC, VEC>(G, objects, h, st, logits, gstart, U, w, args...);
    default: return launch_close<4, RC, VEC>(G, objects, h, st, logits, gstart, U, w, args...);
    }
}

extern "C" rs3_status rs3_close_argmax(const float *logits, const int32_t *group_start, int G, int U, int h,
                                       int w, int radius, int s, uint8_t *palette, uint8_t *closed,
                                       uint8_t *grid_masks, int32_t *status, rs3_stream_t stream)
{
    if (!logits || !group_start || !status) return RS3_EINVAL;
    if (G < 1 || U < 0 || h < 1 || w < 32 || radius < 0 || s < 1) return RS3_EINVAL;
    if (w % 32 != 0 || radius > CA_RMAX) return RS3_EUNSUPPORTED;
    if (grid_masks && (h % s != 0 || w % s != 0)) return RS3_EINVAL;
    if ((long long)h * w > (1ll << 31)) return RS3_EUNSUPPORTED;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // objects of a stream on average, at most 8 (the portable cluster size);
    // ranks past a stream's object count idle
    const int objects = std::min(CA_KCMAX, std::max(1, (U + G - 1) / G));
    if ((long long)G * objects > 65535) return RS3_EUNSUPPORTED;
    // 16-byte loads and 4-byte stores where the arrays allow them
    const auto low = [](const void *p) { return reinterpret_cast<uintptr_t>(p); };
    const bool vec = rs3_aligned16(logits) && ((low(palette) | low(closed)) & 3u) == 0;
    // the paper's 9 x 9 element has kernels of its own; those of a radius at run
    // time take twice the registers, one CTA per SM
    const auto launch = radius == 4 ? (vec ? launch_close_strips<4, true, int, int, uint8_t *, uint8_t *, uint8_t *, int32_t *>
                                           : launch_close_strips<4, false, int, int, uint8_t *, uint8_t *, uint8_t *, int32_t *>)
                                    : (vec ? launch_close_strips<0, true, int, int, uint8_t *, uint8_t *, uint8_t *, int32_t *>
                                           : launch_close_strips<0, false, int, int, uint8_t *, uint8_t *, uint8_t *, int32_t *>);
    const cudaError_t e = launch(G, objects, h, st, logits, group_start, U, w, radius, s, palette, closed, grid_masks, status);
    return e == cudaSuccess ? RS3_OK : RS3_ECUDA;
}

extern "C" rs3_status rs3_seed_from_masks(const uint8_t *masks, int U, int h, int w, int s, rs3_track *track,
                                          uint8_t *grid_masks, uint8_t *box_masks, rs3_stream_t stream)
{
    if (!masks || !track) return RS3_EINVAL;
    if (U < 1 || h < 1 || w < 16 || s < 1) return RS3_EINVAL;
    if (w % 16 != 0 || !rs3_aligned16(masks)) return RS3_EINVAL;
    if (h % s != 0 || w % s != 0) return RS3_EINVAL;
    if (U > 65535) return RS3_EUNSUPPORTED;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    SeedDims d;
    d.h = h; d.w = w; d.s = s; d.m = h / s; d.n = w / s;
    d.cpr = (uint32_t)w / 16;
    const long long chunks = (long long)h * d.cpr, cells = (long long)d.m * d.n;
    // Over all SMs, in three launches, past 1 MB a mask or 16 MB in all (us per call
    // in a graph, cluster and bands; called eagerly the three launches take 11.5 and
    // the one 8 or its own time): 1 x 1024 x 1024 8.2 and 5.0, 1 x 1080 x 1920 11.6 and
    // 5.0, 1 x 4096 x 4096 72 and 8, 16 x 1024 x 1024 10.8 and 8.2, 48 x 384 x 384 5.6
    // and 6.1, 100 x 512 x 512 9.9 and 11.3, 48 x 1024 x 1024 17.8 and 14.7.
    if (chunks > 65536 || U * chunks >= 1 << 20) {
        d.rows = (int)std::min((long long)h, std::max(1ll, SCAN_CHUNKS / (long long)d.cpr));
        d.dx = SCAN_THREADS % d.cpr;
        d.share = 4 * SCAN_THREADS;
        cudaError_t e = launch_pdl(k_seed_init, dim3((U + 255) / 256), dim3(256), 0, st, track, U);
        if (e == cudaSuccess)
            e = launch_pdl(k_seed_scan, dim3((h + d.rows - 1) / d.rows, U), dim3(SCAN_THREADS), 0, st, masks, d, track,
                           grid_masks);
        if (e == cudaSuccess)
            e = launch_pdl(k_seed_finish, dim3(box_masks ? (unsigned)((cells + d.share - 1) / d.share) : 1u, U),
                           dim3(SCAN_THREADS), 0, st, d, track, box_masks);
        return e == cudaSuccess ? RS3_OK : RS3_ECUDA;
    }
    // Threads per unit: as many as load it in one batch of each, but no more than
    // are resident at once (1024 per SM by their registers).
    const long long want = std::max(256ll, std::min((chunks + SEED_BATCH - 1) / SEED_BATCH, 1024ll * rs3_sm_count() / U));
    const int threads = want <= 128 * SEED_KC ? 256 : 512;
    const int KC = (int)std::min((long long)SEED_KC, (want + threads - 1) / threads);
    d.rows = (h + KC - 1) / KC;
    d.dx = (uint32_t)threads % d.cpr;
    d.share = (uint32_t)((cells + KC - 1) / KC);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(KC, U);
    cfg.blockDim = dim3(threads);
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
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_seed, masks, d, KC, track, grid_masks, box_masks);
    return e == cudaSuccess ? RS3_OK : RS3_ECUDA;
}
