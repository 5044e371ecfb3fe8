// rs3_readout_common.cuh -- argument block and helpers shared by the readout
// kernels (CUDA-core and tensor-core paths).
#pragma once

#include "rs3_internal.cuh"

#define RS3_MAX_UNITS 4096  // units per readout call
#define RS3_PAIR_ITEMS (1 << 30)   // above every item index

struct ReadoutArgs {
    const void *q;
    const void *k_store;
    const void *v_store;
    const int64_t *meta;
    int64_t meta_stride_words;
    int64_t pinned_cap, ring_cap, rows_per_unit;
    int64_t n_ptr;
    const int32_t *unit_group;
    const int32_t *idx;
    const int32_t *count;
    const float *rope;
    const void *residual;
    void *out;
    int32_t *status;
    int U, G, mn, H, d, D, k_max;
    int BM, BN, n_sm, min_chunk;
    int plan_ov;            // leading plan slots per group: a piece's start-up cost in tiles
    int either;             // the plan may take the two-tile kernel (the four above are the one-tile kernel's)
    int tensor;             // a tensor-core kernel runs the plan
    int64_t max_slots;
    int grid_ctas;          // CTAs of the readout launch (the plan's slice count bound)
    int32_t *cta_items;     // [grid_ctas][2]: CTA b runs items [cta_items[2b], cta_items[2b+1]); the first
                            // of the two with RS3_PAIR_ITEMS where they are for the two-tile kernel
    float scale_log2;       // softmax scale * log2(e)
    uint64_t wait_ns;       // limit of each device-side wait (global-timer ns)
    ReadoutHeader *header;
    RangeSet *ranges;
    WorkItem *items;
    CombineItem *combine;
    float *part_o;          // [slot][BM][d]
    float *part_ml;         // [slot][BM] (m, l) pairs, m in the log2 domain
};

struct ReadoutPath {
    int kind;        // 0 = CUDA-core, 1 = tensor-core (tcgen05)
    bool either;     // ... with one or two query tiles, as the plan finds
    int BM, BN;      // of one query tile
    int part_rows;   // rows of a partial slot
    int grid;   // CTAs of the readout launch
};

// the path of a call over banks of this many rows with this workspace (INT64_MAX and
// SIZE_MAX: the path that any workspace is sized for)
ReadoutPath choose_readout_path(rs3_dtype dtype, int d, int U, int H, int k_max, int64_t bank_rows, size_t workspace_bytes);
bool rs3_tc_supported(int d);
int rs3_tc_block_n(int d);
rs3_status rs3_launch_tc_readout(const ReadoutArgs &a, cudaStream_t st);
rs3_status rs3_launch_either_readout(const ReadoutArgs &a, cudaStream_t st);   // d = 64, 128
// CUDA-core path: rows and keys of a tile and resident CTAs per SM, for a head width
void rs3_simt_tile(int d, int &bm, int &bn, int &ctas_per_sm);
rs3_status rs3_launch_simt_readout(const ReadoutArgs &a, rs3_dtype dtype, cudaStream_t st);
rs3_status rs3_readout_prepare(const void *q, rs3_dtype dtype, int G, int mn, int H, int d,
                               const int32_t *unit_group, const int32_t *idx, const int32_t *count,
                               int k_max, const rs3_bank *bank, const float *rope,
                               const void *residual, void *out, float scale, void *workspace,
                               size_t workspace_bytes, int32_t *status, ReadoutArgs *a,
                               ReadoutPath *path, int64_t *grid_combine);
// phases of a readout: the attention over the bank (pass-through, plan,
// readout kernel) and the merge of split-KV partials
enum { RS3_PHASE_PLAN = 1, RS3_PHASE_RUN = 4, RS3_PHASE_ATTEND = 1 | 4, RS3_PHASE_MERGE = 2 };
rs3_status rs3_readout_launch(const ReadoutArgs &a, const ReadoutPath &p,
                              int64_t max_combine, rs3_dtype dtype, cudaStream_t st, int phases);

// Tile t of a unit's bank (tiles of BN rows, never crossing a range end) ->
// first physical row and the number of valid rows.
__device__ __forceinline__ void tile_rows(const RangeSet &rs, int t, int BN, int64_t &row0, int &nvalid)
{
    row0 = 0;
    nvalid = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        if (t < rs.tiles[r]) {
            row0 = rs.start[r] + (int64_t)t * BN;
            nvalid = min(BN, rs.len[r] - t * BN);
            return;
        }
        t -= rs.tiles[r];
    }
}

// Same, reading the range set in place (global memory) instead of a local copy.
__device__ __forceinline__ void tile_rows(const RangeSet *rs, int t, int BN, int64_t &row0, int &nvalid)
{
    row0 = 0;
    nvalid = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int tiles = __ldg(&rs->tiles[r]);
        if (t < tiles) {
            row0 = __ldg(&rs->start[r]) + (int64_t)t * BN;
            nvalid = min(BN, __ldg(&rs->len[r]) - t * BN);
            return;
        }
        t -= tiles;
    }
}

__device__ __forceinline__ float4 load4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ float4 load4(const uint16_t *p)
{
    const uint2 w = __ldg(reinterpret_cast<const uint2 *>(p));
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                       __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
}

// Two fp32 values to a bf16 pair (round to nearest even), `lo` in the low half;
// one cvt instruction (the per-value conversions cost about three times more).
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// A 16-byte piece of a query row (four pairs) rotated by the (cos, sin) of those
// pairs at f (Eq. 7), rounded once per element.
__device__ __forceinline__ uint4 rotate_q_piece(uint4 v, const float *f)
{
    uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int p = 0; p < 4; p += 2) {
        const float4 c = __ldg(reinterpret_cast<const float4 *>(f) + p / 2);
        const float x0 = __uint_as_float(w[p] << 16), x1 = __uint_as_float(w[p] & 0xffff0000u);
        const float y0 = __uint_as_float(w[p + 1] << 16), y1 = __uint_as_float(w[p + 1] & 0xffff0000u);
        w[p] = pack_bf16x2(x0 * c.x - x1 * c.y, x0 * c.y + x1 * c.x);
        w[p + 1] = pack_bf16x2(y0 * c.z - y1 * c.w, y0 * c.w + y1 * c.z);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// out[u][cell][c .. c+1] (store_out2) or [c .. c+3] (store_out4) =
// residual[...] + o, rounded once to T
template <typename T>
__device__ __forceinline__ void store_out2(const ReadoutArgs &a, int u, int cell, int c, const float *o);

template <>
__device__ __forceinline__ void store_out2<float>(const ReadoutArgs &a, int u, int cell, int c, const float *o)
{
    const int64_t off = ((int64_t)u * a.mn + cell) * a.D + c;
    float2 r = make_float2(0.f, 0.f);
    if (a.residual) r = *reinterpret_cast<const float2 *>(static_cast<const float *>(a.residual) + off);
    *reinterpret_cast<float2 *>(static_cast<float *>(a.out) + off) = make_float2(r.x + o[0], r.y + o[1]);
}

template <>
__device__ __forceinline__ void store_out2<uint16_t>(const ReadoutArgs &a, int u, int cell, int c, const float *o)
{
    const int64_t off = ((int64_t)u * a.mn + cell) * a.D + c;
    float r0 = 0.f, r1 = 0.f;
    if (a.residual) {
        const uint32_t x = *reinterpret_cast<const uint32_t *>(static_cast<const uint16_t *>(a.residual) + off);
        r0 = __uint_as_float(x << 16);
        r1 = __uint_as_float(x & 0xffff0000u);
    }
    *reinterpret_cast<uint32_t *>(static_cast<uint16_t *>(a.out) + off) = pack_bf16x2(r0 + o[0], r1 + o[1]);
}

template <typename T>
__device__ __forceinline__ void store_out4(const ReadoutArgs &a, int u, int cell, int c, const float *o);

template <>
__device__ __forceinline__ void store_out4<float>(const ReadoutArgs &a, int u, int cell, int c, const float *o)
{
    const int64_t off = ((int64_t)u * a.mn + cell) * a.D + c;
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.residual) r = load4(static_cast<const float *>(a.residual) + off);
    *reinterpret_cast<float4 *>(static_cast<float *>(a.out) + off) =
        make_float4(r.x + o[0], r.y + o[1], r.z + o[2], r.w + o[3]);
}

template <>
__device__ __forceinline__ void store_out4<uint16_t>(const ReadoutArgs &a, int u, int cell, int c, const float *o)
{
    const int64_t off = ((int64_t)u * a.mn + cell) * a.D + c;
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.residual) r = load4(static_cast<const uint16_t *>(a.residual) + off);
    *reinterpret_cast<uint2 *>(static_cast<uint16_t *>(a.out) + off) =
        make_uint2(pack_bf16x2(r.x + o[0], r.y + o[1]), pack_bf16x2(r.z + o[2], r.w + o[3]));
}
