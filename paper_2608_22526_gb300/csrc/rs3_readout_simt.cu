// rs3_readout_simt.cu -- CUDA-core flash readout (Sec. 3.1, Eq. 6 and Eq. 7):
// fp32 at every head width, bf16 where the tensor-core path has no tile
// (d = 16, 32).  All products and sums are fp32.
//
// It is bound by the fp32 FMA pipe, so both contractions are register-tiled
// and run on packed pairs (fma.rn.f32x2).  A CTA of four warps takes BM query
// rows; a warp owns RW = 4 TM of them for the whole item, so the softmax needs
// no exchange between warps and P never leaves the warp.  Lane (tr, tk) =
// (lane / 8, lane % 8) holds rows 4 i + tr and, of the 32 keys of a tile, keys
// tk + 8 j:
//   S = Q K^T   accumulator pairs run along d (even and odd sums, added once),
//               so both operands are read as they lie in memory: TM + 4
//               16-byte shared loads feed 8 TM packed FMAs;
//   O += P V    accumulator pairs run along the output columns: a 16-byte
//               load of P is four keys of a row, each doubled by a move.
// Rows in shared memory are padded by 16 bytes, which puts the four rows and
// the eight keys of a warp's load on different banks.  Tiles of 32 keys are
// double-buffered with cp.async (one barrier per tile).
// One object, 64 x 64 grid, 4 heads of 64, about 7 600 keys (9.6 GFLOP):
// 220 us for the call, 43.6 TFLOP/s of the pipe's 77.8 (1 109 us with one
// row's dot products spread over d / 16 lanes and summed by shuffles).  The
// rest is the softmax's instructions and, with two warps per scheduler (the
// accumulators fill the register file), waits on shared memory.  Lanes that
// share an operand sit next to each other (tk in lane bits 1..3): with tk in
// the low bits a key load took four shared-memory passes instead of two, and
// P stored twice per value in place of a move per value doubled its loads;
// together 260 us.
#include "rs3_readout_common.cuh"
#include "rs3_tc_ptx.cuh"

namespace {

constexpr int BN = 32;              // keys per tile
constexpr int NW = 4;               // warps per CTA

template <int D>
struct Cfg {
    static constexpr int TM = D <= 128 ? 8 : 4;      // rows per lane
    static constexpr int RW = 4 * TM;                // rows per warp
    static constexpr int BM = NW * RW;
    static constexpr int LD = D + 4;                 // row stride in shared memory (floats)
    static constexpr int PLD = BN + 8;               // row stride of P
    // Columns per partial sum of S.  Heads of 64 in one chain: error against 64
    // bits 5.6e-7 of the largest output, 4.4e-7 like this, at 2% of the time.
    static constexpr int KC = D == 256 ? 16 : D < 32 ? D : 32;
    static constexpr int KG = D <= 128 ? D : 128;    // columns per group of partial sums
    static constexpr int TC = D / 8;                 // output columns per lane
    static constexpr int VW = TC < 4 ? TC : 4;       // columns per load
    static constexpr int NJ = TC / VW;
    static constexpr int SMEM = 4 * (BM * LD + 2 * 2 * BN * LD + BM * PLD);
    static constexpr int CTAS = SMEM <= 113 * 1024 ? 2 : 1;   // resident per SM
};

using tc::fma2;
using tc::mul2;

__device__ __forceinline__ void cp_async16(float *dst, const float *src, bool in)
{
    // `in` false writes zeros (nothing is read)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// One tile of K and V rows into shared memory as fp32, zeros past nvalid.
// Thread x copies 16 bytes (of fp32) at column c4 of rows r0, r0 + RPP, ...
template <int D>
struct Stage {
    static constexpr int VPR = D / 4, RPP = NW * 32 / VPR, N = BN / RPP;
    static_assert(NW * 32 % VPR == 0 && BN % RPP == 0, "whole passes");
    int r0, c4;
    __device__ Stage() : r0(threadIdx.x / VPR), c4(threadIdx.x % VPR * 4) {}
    __device__ __forceinline__ void operator()(float *sK, float *sV, const float *K, const float *V, int64_t stride,
                                               int nvalid) const
    {
        const int64_t off = r0 * stride + c4;
        const float *k = K + off, *v = V + off;
        float *dk = sK + r0 * Cfg<D>::LD + c4, *dv = sV + r0 * Cfg<D>::LD + c4;
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const bool in = r0 + n * RPP < nvalid;
            cp_async16(dk + n * RPP * Cfg<D>::LD, in ? k : K, in);
            cp_async16(dv + n * RPP * Cfg<D>::LD, in ? v : V, in);
            k += RPP * stride;
            v += RPP * stride;
        }
    }
    __device__ __forceinline__ void operator()(float *sK, float *sV, const uint16_t *K, const uint16_t *V,
                                               int64_t stride, int nvalid) const
    {
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const int kk = r0 + n * RPP;
            float4 kv = make_float4(0.f, 0.f, 0.f, 0.f), vv = kv;
            if (kk < nvalid) {
                kv = load4(K + kk * stride + c4);
                vv = load4(V + kk * stride + c4);
            }
            *reinterpret_cast<float4 *>(sK + kk * Cfg<D>::LD + c4) = kv;
            *reinterpret_cast<float4 *>(sV + kk * Cfg<D>::LD + c4) = vv;
        }
    }
};

// A unit's ranges in registers: tile t's first row and valid rows.
struct Tiles {
    int64_t start[4];
    int32_t len[4], tiles[4];
    __device__ __forceinline__ explicit Tiles(const RangeSet *rs)
    {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            start[r] = __ldg(&rs->start[r]);
            len[r] = __ldg(&rs->len[r]);
            tiles[r] = __ldg(&rs->tiles[r]);
        }
    }
    __device__ __forceinline__ int64_t row(int t, int &nvalid) const
    {
        int64_t row0 = 0;
        nvalid = 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (t >= 0 && t < tiles[r]) {
                row0 = start[r] + (int64_t)t * BN;
                nvalid = min(BN, len[r] - t * BN);
            }
            t -= tiles[r];
        }
        return row0;
    }
};

template <typename T, int D>
__global__ void __launch_bounds__(NW * 32, Cfg<D>::CTAS) k_readout_simt(ReadoutArgs a)
{
    using C = Cfg<D>;
    constexpr int TM = C::TM, RW = C::RW, BM = C::BM, LD = C::LD, PLD = C::PLD, KC = C::KC, KG = C::KG,
                  TC = C::TC, VW = C::VW, NJ = C::NJ;
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tr = (lane & 1) | (lane >> 4) << 1,
              tk = lane >> 1 & 7;
    float *sQ = sm + warp * RW * LD;                         // this warp's rows [RW][LD]
    float *sKV = sm + BM * LD;                               // [2][K, V][BN][LD]
    float *sP = sKV + 4 * BN * LD + warp * RW * PLD;         // this warp's P [RW][PLD]
    const Stage<D> stage;
    const int it_end = a.cta_items[2 * blockIdx.x + 1];
    for (int it = a.cta_items[2 * blockIdx.x]; it < it_end; ++it) {
        const WorkItem w = a.items[it];
        const RangeSet *rs = a.ranges + w.u;
        const int g = a.unit_group[w.u];
        if (g < 0 || g >= a.G) {                             // uniform over the CTA
            if (threadIdx.x == 0) latch_status(a.status, RS3_EINVAL);
            continue;
        }
        const int cnt = __ldg(&rs->cnt);
        const T *Kb = static_cast<const T *>(a.k_store) + (int64_t)w.u * a.rows_per_unit * a.D + w.h * D;
        const T *Vb = static_cast<const T *>(a.v_store) + (int64_t)w.u * a.rows_per_unit * a.D + w.h * D;
        __syncthreads();                                     // the previous item's last tile has been read
        const Tiles tiles(rs);
        int nvalid = 0;
        if (w.tile_begin < w.tile_end) {
            const int64_t off = tiles.row(w.tile_begin, nvalid) * a.D;
            stage(sKV, sKV + BN * LD, Kb + off, Vb + off, a.D, nvalid);
        }
        cp_async_commit();
        // the kept query rows, rotated by their own cell and scaled (zeros past
        // the kept count)
        constexpr int QB = RW * D / 128 < 8 ? RW * D / 128 : 8;   // pieces in flight per lane
        for (int e0 = lane; e0 < RW * (D / 4); e0 += 32 * QB) {
            int cell[QB];
            float4 x[QB], f[QB];
#pragma unroll
            for (int n = 0; n < QB; ++n) {
                const int j = w.qt * BM + warp * RW + (e0 + 32 * n) / (D / 4);
                cell[n] = j < cnt ? __ldg(a.idx + (int64_t)w.u * a.k_max + j) : -1;
                if (j < cnt && (cell[n] < 0 || cell[n] >= a.mn)) cell[n] = 0;
            }
#pragma unroll
            for (int n = 0; n < QB; ++n) {
                const int c4 = (e0 + 32 * n) % (D / 4) * 4;
                x[n] = make_float4(0.f, 0.f, 0.f, 0.f);
                f[n] = make_float4(1.f, 0.f, 1.f, 0.f);
                if (cell[n] < 0) continue;
                x[n] = load4(static_cast<const T *>(a.q) + ((int64_t)g * a.mn + cell[n]) * a.D + w.h * D + c4);
                if (a.rope) f[n] = __ldg(reinterpret_cast<const float4 *>(a.rope + (int64_t)cell[n] * D + c4));
            }
#pragma unroll
            for (int n = 0; n < QB; ++n) {
                const int r = (e0 + 32 * n) / (D / 4), c4 = (e0 + 32 * n) % (D / 4) * 4;
                float4 y = x[n];
                if (a.rope)
                    y = make_float4(y.x * f[n].x - y.y * f[n].y, y.x * f[n].y + y.y * f[n].x,
                                    y.z * f[n].z - y.w * f[n].w, y.z * f[n].w + y.w * f[n].z);
                *reinterpret_cast<float4 *>(sQ + r * LD + c4) = make_float4(
                    y.x * a.scale_log2, y.y * a.scale_log2, y.z * a.scale_log2, y.w * a.scale_log2);
            }
        }
        uint64_t o[TM][TC / 2];
        float mrun[TM], lrun[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            mrun[i] = -INFINITY;
            lrun[i] = 0.f;
#pragma unroll
            for (int c = 0; c < TC / 2; ++c) o[i][c] = 0ull;
        }
        __syncwarp();
        for (int t = w.tile_begin; t < w.tile_end; ++t) {
            const int buf = (t - w.tile_begin) & 1;
            const float *sK = sKV + buf * 2 * BN * LD, *sV = sK + BN * LD;
            const int nv = nvalid;
            cp_async_wait();
            __syncthreads();                                 // tile t is in; every warp has read tile t - 1
            if (t + 1 < w.tile_end) {
                const int64_t off = tiles.row(t + 1, nvalid) * a.D;
                float *nK = sKV + (buf ^ 1) * 2 * BN * LD;
                stage(nK, nK + BN * LD, Kb + off, Vb + off, a.D, nvalid);
            }
            cp_async_commit();
            // S = Q K^T, for wide heads in partial sums of KC columns, so that
            // the chains of roundings are no longer than at d = 64
            float s[TM][4];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) s[i][j] = 0.f;
            const float *qp = sQ + tr * LD, *kp = sK + tk * LD;
#pragma unroll 1
            for (int kg = 0; kg < D; kg += KG) {
                float sg[TM][4];
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) sg[i][j] = 0.f;
#pragma unroll 1
                for (int k0 = kg; k0 < kg + KG; k0 += KC) {
                    uint64_t acc[TM][4];
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
#pragma unroll 8
                    for (int k = k0; k < k0 + KC; k += 4) {
                        ulonglong2 kv[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) kv[j] = *reinterpret_cast<const ulonglong2 *>(kp + 8 * j * LD + k);
#pragma unroll
                        for (int i0 = 0; i0 < TM; i0 += 4) {
                            ulonglong2 qv[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                qv[i] = *reinterpret_cast<const ulonglong2 *>(qp + 4 * (i0 + i) * LD + k);
#pragma unroll
                            for (int i = 0; i < 4; ++i)
#pragma unroll
                                for (int j = 0; j < 4; ++j) acc[i0 + i][j] = fma2(qv[i].x, kv[j].x, acc[i0 + i][j]);
#pragma unroll
                            for (int i = 0; i < 4; ++i)
#pragma unroll
                                for (int j = 0; j < 4; ++j) acc[i0 + i][j] = fma2(qv[i].y, kv[j].y, acc[i0 + i][j]);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            float lo, hi;
                            tc::f2unpack(acc[i][j], lo, hi);
                            sg[i][j] = KC == KG ? lo + hi : sg[i][j] + (lo + hi);
                        }
                }
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) s[i][j] = KG == D ? sg[i][j] : s[i][j] + sg[i][j];
            }
            if (nv < BN) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (tk + 8 * j >= nv) {
#pragma unroll
                        for (int i = 0; i < TM; ++i) s[i][j] = -INFINITY;
                    }
            }
            // The reference of a row's exps moves only when a score passes it by
            // more than 2^8 (and at the first tile): values up to 2^8 lose
            // nothing in fp32, and most tiles need no reduction over the lanes.
            bool grow = false;
#pragma unroll
            for (int i = 0; i < TM; ++i)
                grow |= !(fmaxf(fmaxf(s[i][0], s[i][1]), fmaxf(s[i][2], s[i][3])) <= mrun[i] + 8.0f);
            if (__any_sync(0xffffffffu, grow)) {
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    float mt = fmaxf(fmaxf(s[i][0], s[i][1]), fmaxf(s[i][2], s[i][3]));
#pragma unroll
                    for (int off = 8; off >= 2; off >>= 1) mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, off));
                    const float mnew = fmaxf(mrun[i], mt);
                    const float alpha = exp2f(mrun[i] - mnew);
                    const uint64_t al2 = tc::f2pack(alpha, alpha);
                    lrun[i] *= alpha;
#pragma unroll
                    for (int c = 0; c < TC / 2; ++c) o[i][c] = mul2(o[i][c], al2);
                    mrun[i] = mnew;
                }
            }
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float p = tc::ex2_approx(s[i][j] - mrun[i]);
                    lrun[i] += p;
                    sP[(4 * i + tr) * PLD + tk + 8 * j] = p;
                }
            __syncwarp();
            // O += P V.  Heads of 256 sum a tile's keys first (JG loads of columns at
            // a time) and add the sums: with one CTA per SM their work items hold the
            // longest runs of keys.  80 x 80 grid, flat scores: error 2.4e-7 of the
            // largest output, 5.8e-7 in one chain, for 2% of the time.
            const float *pp = sP + tr * PLD, *vp = sV + tk * VW;
            constexpr int JG = D == 256 ? 4 : NJ, CG = JG * VW / 2;
#pragma unroll
            for (int j0 = 0; j0 < NJ; j0 += JG) {
                uint64_t t[TM][CG];
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int c = 0; c < CG; ++c) t[i][c] = JG == NJ ? o[i][c] : 0ull;
#pragma unroll 2
                for (int k = 0; k < BN; k += 4) {
                    float4 p[TM];
#pragma unroll
                    for (int i = 0; i < TM; ++i) p[i] = *reinterpret_cast<const float4 *>(pp + 4 * i * PLD + k);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        uint64_t v[CG];
#pragma unroll
                        for (int j = 0; j < JG; ++j) {
                            if constexpr (VW == 4) {
                                const ulonglong2 x =
                                    *reinterpret_cast<const ulonglong2 *>(vp + (k + kk) * LD + 32 * (j0 + j));
                                v[2 * j] = x.x;
                                v[2 * j + 1] = x.y;
                            } else {
                                v[j] = *reinterpret_cast<const uint64_t *>(vp + (k + kk) * LD);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < TM; ++i) {
                            const float pk = kk == 0 ? p[i].x : kk == 1 ? p[i].y : kk == 2 ? p[i].z : p[i].w;
                            const uint64_t p2 = tc::f2pack(pk, pk);
#pragma unroll
                            for (int c = 0; c < CG; ++c) t[i][c] = fma2(p2, v[c], t[i][c]);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int c = 0; c < CG; ++c) {
                        uint64_t &oc = o[i][j0 * VW / 2 + c];
                        oc = JG == NJ ? t[i][c] : tc::add2(oc, t[i][c]);
                    }
            }
            __syncwarp();                                    // P is read before the next tile's is written
        }
        // epilogue: residual + O / l at the kept cell, or the split-KV partial
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            float l = lrun[i];
#pragma unroll
            for (int off = 8; off >= 2; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
            const int r = warp * RW + 4 * i + tr, j = w.qt * BM + r;
            if (j >= cnt) continue;
            float x[TC];
#pragma unroll
            for (int c = 0; c < TC / 2; ++c) tc::f2unpack(o[i][c], x[2 * c], x[2 * c + 1]);
            if (w.slot < 0) {
                const float inv = l > 0.f ? 1.f / l : 0.f;
                int cell = a.idx[(int64_t)w.u * a.k_max + j];
                if (cell < 0 || cell >= a.mn) cell = 0;
#pragma unroll
                for (int n = 0; n < TC; ++n) x[n] *= inv;
#pragma unroll
                for (int n = 0; n < NJ; ++n) {
                    const int c0 = w.h * D + 32 * n + tk * VW;
                    if constexpr (VW == 4) store_out4<T>(a, w.u, cell, c0, x + 4 * n);
                    else store_out2<T>(a, w.u, cell, c0, x);
                }
            } else {
                float *po = a.part_o + ((int64_t)w.slot * BM + r) * D + tk * VW;
#pragma unroll
                for (int n = 0; n < NJ; ++n) {
                    if constexpr (VW == 4)
                        *reinterpret_cast<float4 *>(po + 32 * n) =
                            make_float4(x[4 * n], x[4 * n + 1], x[4 * n + 2], x[4 * n + 3]);
                    else
                        *reinterpret_cast<float2 *>(po) = make_float2(x[0], x[1]);
                }
                if (tk == 0)
                    reinterpret_cast<float2 *>(a.part_ml)[(int64_t)w.slot * BM + r] = make_float2(mrun[i], l);
            }
        }
    }
}

template <typename T, int D>
rs3_status launch(const ReadoutArgs &a, cudaStream_t st)
{
    if (rs3_kernel_smem((const void *)k_readout_simt<T, D>, Cfg<D>::SMEM) != RS3_OK) return RS3_ECUDA;
    launch_pdl(k_readout_simt<T, D>, dim3((unsigned)a.grid_ctas), dim3(NW * 32), Cfg<D>::SMEM, st, a);
    return cudaGetLastError() == cudaSuccess ? RS3_OK : RS3_ECUDA;
}

}  // namespace

void rs3_simt_tile(int d, int &bm, int &bn, int &ctas_per_sm)
{
    bn = BN;
    switch (d) {
    case 16: bm = Cfg<16>::BM; ctas_per_sm = Cfg<16>::CTAS; break;
    case 32: bm = Cfg<32>::BM; ctas_per_sm = Cfg<32>::CTAS; break;
    case 64: bm = Cfg<64>::BM; ctas_per_sm = Cfg<64>::CTAS; break;
    case 128: bm = Cfg<128>::BM; ctas_per_sm = Cfg<128>::CTAS; break;
    default: bm = Cfg<256>::BM; ctas_per_sm = Cfg<256>::CTAS; break;
    }
}

rs3_status rs3_launch_simt_readout(const ReadoutArgs &a, rs3_dtype dtype, cudaStream_t st)
{
    if (dtype == RS3_BF16) {                 // the other widths have a tensor-core tile
        switch (a.d) {
        case 16: return launch<uint16_t, 16>(a, st);
        case 32: return launch<uint16_t, 32>(a, st);
        default: return RS3_EUNSUPPORTED;
        }
    }
    switch (a.d) {
    case 16: return launch<float, 16>(a, st);
    case 32: return launch<float, 32>(a, st);
    case 64: return launch<float, 64>(a, st);
    case 128: return launch<float, 128>(a, st);
    case 256: return launch<float, 256>(a, st);
    default: return RS3_EUNSUPPORTED;
    }
}
