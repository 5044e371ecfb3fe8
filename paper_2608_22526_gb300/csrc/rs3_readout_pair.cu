// rs3_readout_pair.cu -- tensor-core readout for bf16 heads of 64 and 128
// (Sec. 3.1, Eq. 6 and Eq. 7) on sm_103a: two query tiles per CTA.
//
// At these widths a 128 x 128 tile of scores costs the exponentials as much
// time as the tensor core (d = 64: 512 clk each), so the softmax must never
// wait for the matrices nor they for it.  A work item is 256 kept queries, two
// tiles of 128 that share the K and V tiles; each tile has its own S in TMEM
// and its own softmax warpgroup, a thread per row: no exchange between threads,
// and while one warpgroup takes its exps the tensor core works for the other.
//   warp 0      TMA of K and V tiles (128 keys) into two rings
//   warps 1, 2  issue query tile 0's (1's) S_q = Q_q K^T (both operands in
//               shared memory) and O_q += P_q V (P_q in TMEM)
//   warps 4-7   softmax of query tile 0, warps 8-11 of tile 1: per item the
//               kept rows (rotated by the RoPE table of their own cell) into
//               shared memory; per tile the row's 128 scores into registers,
//               exps against a running reference that moves only when a score
//               passes it by 2^8, P_q to TMEM as bf16 pairs; epilogue O / l +
//               residual, or the split-KV partial.  The next item's query rows
//               are loaded before the epilogue, while the last P V runs.
// An item of at most 128 rows uses tile 0 alone.
//
// What is faster depends on the kept queries and the banks' lengths, which only the
// device knows, so k_readout_either holds this kernel and the one-tile one
// (rs3_readout_tc.cuh) on the same threads, and the plan marks the item ranges with
// its choice.  Chosen by k_max on the host, 3 objects of 2 heads of 128 with 300 kept
// queries and 600 keys each took 26.9 us; 16.6 with one tile, 18.2 before.  The tc
// kernel's start is up to 1.8 us slower inside the larger kernel.
// TMEM: d = 64: O_0, O_1, S_0, S_1 and P_0, P_1 fill the 512 columns, so
// S_q(t + 1) needs only that S_q(t) was read.  d = 128: P_q lies over S_q, and
// S_q(t + 1) is issued behind the P V that reads it (the tensor core takes a
// CTA's matrix instructions in order).
// The softmax warps take registers from the others (setmaxnreg): a row's 128
// scores stay in registers.
// 16 streams x 3 objects, 4 heads of 64, 96 x 96 grid (911 GFLOP): 1 078 us per
// call, 1 704 in the one-tile kernel.  Per pair of 128 x 128 tiles it takes about
// 2 500 clk, where the exps of 256 rows alone take 1 380 and the matrices 1 052:
// a warpgroup's own chain (wait, scores from TMEM, max, exps, P to TMEM) is that
// long with two warps per scheduler.
// Every mbarrier wait is bounded as in rs3_readout_tc.cuh.
#include "rs3_readout_tc.cuh"

namespace tc {

namespace pair {

constexpr int BQ = 128;             // rows of a query tile
constexpr int BN = 128;             // keys per tile
constexpr uint32_t TMEM_COLS = 512;
constexpr int NTHREADS = 384;

template <int DH>
struct Cfg {
    static constexpr int KVBYTES = BN * DH * 2;              // one K (or V) stage
    static constexpr int QBYTES = BQ * DH * 2;               // one query tile
    static constexpr int NKV = (232448 - 1024 - 512 - 2 * QBYTES) / KVBYTES;
    static constexpr int KSTK = (NKV + 1) / 2, KSTV = NKV / 2;
    static constexpr bool PSEP = DH == 64;                   // P beside S instead of over it
    static constexpr uint32_t O_COL = 0, S_COL = 2 * DH, P_COL = PSEP ? 2 * DH + 2 * BN : S_COL;
    static constexpr uint32_t P_STEP = PSEP ? BN / 2 : BN;   // columns between P_0 and P_1
    // registers after the split; the launch has 168 for each of 3 x 128 threads
    static constexpr int REGS_ISSUE = 88, REGS_SOFTMAX = 208;
    static_assert(REGS_ISSUE + 2 * REGS_SOFTMAX <= 3 * 168, "register split");
    static constexpr int OFF_Q = 0;
    static constexpr int OFF_K = OFF_Q + 2 * QBYTES;
    static constexpr int OFF_V = OFF_K + KSTK * KVBYTES;
    static constexpr int OFF_BAR = OFF_V + KSTV * KVBYTES;
    // barriers: the rings, then per query tile
    static constexpr int B_KFULL = 0, B_KEMPTY = KSTK, B_VFULL = 2 * KSTK, B_VEMPTY = 2 * KSTK + KSTV;
    static constexpr int B_QFULL = 2 * KSTK + 2 * KSTV, B_SFULL = B_QFULL + 2, B_SFREE = B_QFULL + 4;
    static constexpr int B_PFULL = B_QFULL + 6, B_PVDONE = B_QFULL + 8, B_OFREE = B_QFULL + 10;
    static constexpr int B_DRAIN = B_QFULL + 12, NBAR = B_QFULL + 13;
    static constexpr int OFF_MISC = OFF_BAR + NBAR * 8;
    static constexpr int SMEM = OFF_MISC + 16 + 1024;        // + alignment slack
    static_assert(S_COL + 2 * BN <= TMEM_COLS && P_COL + P_STEP + BN / 2 <= TMEM_COLS, "TMEM budget");
    static_assert(KSTK >= 2 && KSTV >= 2 && SMEM <= 232448 && NBAR * 8 + 16 <= 512, "shared memory budget");
};

template <int N>
__device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

// The kept query row of this thread (one row of a tile) into shared memory,
// K-major and 128-byte swizzled; zeros past the kept count (qrow null).
template <int DH>
__device__ __forceinline__ void store_q_row(uint32_t sq, int r, const uint16_t *qrow, const float *rope)
{
#pragma unroll
    for (int c0 = 0; c0 < DH / 8; c0 += 8) {
        uint4 v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c)
            v[c] = qrow ? __ldg(reinterpret_cast<const uint4 *>(qrow) + c0 + c) : make_uint4(0u, 0u, 0u, 0u);
        if (qrow && rope) {
#pragma unroll
            for (int c = 0; c < 8; ++c) v[c] = rotate_q_piece(v[c], rope + 8 * (c0 + c));
        }
#pragma unroll
        for (int c = 0; c < 8; ++c)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(sq + sw128_offset(BQ, r, c0 + c)), "r"(v[c].x),
                         "r"(v[c].y), "r"(v[c].z), "r"(v[c].w) : "memory");
    }
}

// The tile ranges of a unit's bank, walked tile by tile: the valid rows of the
// next tile (a tile never crosses a range's end).
struct TileWalk {
    int rem, k, len[4];
    __device__ __forceinline__ TileWalk(const RangeSet *rs, int tile)
    {
        k = 0;
        rem = 0;
        int t = tile;
#pragma unroll
        for (int r = 0; r < 4; ++r) len[r] = __ldg(&rs->len[r]);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int tiles = (len[r] + BN - 1) / BN;
            if (t >= 0 && t < tiles) {
                k = r;
                rem = len[r] - t * BN;
            }
            t -= tiles;
        }
    }
    __device__ __forceinline__ int next()
    {
        if (rem <= 0) {
#pragma unroll
            for (int r = 1; r < 4; ++r)
                if (r > k && rem <= 0) {
                    rem = len[r];
                    k = r;
                }
        }
        const int nv = min(BN, rem);
        rem -= BN;
        return nv;
    }
};

// Items [it_begin, it_end) of the plan, in a CTA that is set up for the one-tile
// kernel (set_up_tc): its tensor memory serves, its barriers make room.
template <int DH>
__device__ __forceinline__ void readout_pair(const ReadoutArgs &a, const CUtensorMap &tmk, const CUtensorMap &tmv,
                                             uint32_t tmem, int it_begin, int it_end)
{
    using C = Cfg<DH>;
    constexpr int KSTK = C::KSTK, KSTV = C::KSTV;
    static_assert(TMEM_COLS == tc::TMEM_COLS, "one allocation for both kernels");
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *gbase = smem_raw + (base - raw);
    const uint32_t sQ = base + C::OFF_Q, sK = base + C::OFF_K, sV = base + C::OFF_V;
    const uint32_t bars = base + C::OFF_BAR;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(gbase + C::OFF_MISC);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#define BAR(i) (bars + 8u * (uint32_t)(i))

    if (threadIdx.x == 0) {
        for (int i = 0; i < tc::Cfg<DH>::NBAR; ++i) mbar_inval(base + tc::Cfg<DH>::OFF_BAR + 8u * i);
        for (int s = 0; s < KSTK; ++s) {
            mbar_init(BAR(C::B_KFULL + s), 1);
            mbar_init(BAR(C::B_KEMPTY + s), 2);               // both MMA issuers
        }
        for (int s = 0; s < KSTV; ++s) {
            mbar_init(BAR(C::B_VFULL + s), 1);
            mbar_init(BAR(C::B_VEMPTY + s), 2);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(BAR(C::B_QFULL + q), 4);                // one arrival per softmax warp
            mbar_init(BAR(C::B_SFULL + q), 1);
            mbar_init(BAR(C::B_SFREE + q), 4);
            mbar_init(BAR(C::B_PFULL + q), 4);
            mbar_init(BAR(C::B_PVDONE + q), 1);
            mbar_init(BAR(C::B_OFREE + q), 4);
        }
        mbar_init(BAR(C::B_DRAIN), 2);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    __syncthreads();
    const uint64_t wait_ns = a.wait_ns;

    if (warp < 4) {
        reg_dec<C::REGS_ISSUE>();
        if (warp == 0 && lane == 0) {
            // ------------------------------------------------------------------
            // TMA producer: tile t's K, then tile t's V
            // ------------------------------------------------------------------
            constexpr int BOX = tc::Cfg<DH>::BN;                       // rows of the one-tile kernel's boxes
            uint32_t ck = 0, cv = 0;                                   // K and V tiles issued
            bool ok = true;
            for (int it = it_begin; it < it_end && ok; ++it) {
                const WorkItem w = a.items[it];
                const RangeSet *rs = a.ranges + w.u;
                for (int t = w.tile_begin; t < w.tile_end; ++t) {
                    int64_t row0;
                    int nvalid;
                    tile_rows(rs, t, BN, row0, nvalid);
                    const int y = (int)((int64_t)w.u * a.rows_per_unit + row0);
                    const uint32_t ks = ck % KSTK, vs = cv % KSTV;
                    ok = mbar_wait(BAR(C::B_KEMPTY + ks), ((ck / KSTK) & 1u) ^ 1u, abort_flag, wait_ns);
                    if (!ok) break;
                    mbar_expect_tx(BAR(C::B_KFULL + ks), (uint32_t)C::KVBYTES);
#pragma unroll
                    for (int c = 0; c < DH / 64; ++c)
#pragma unroll
                        for (int r = 0; r < BN; r += BOX)
                            tma_load_2d(sK + ks * C::KVBYTES + c * (BN * 128) + r * 128, &tmk, BAR(C::B_KFULL + ks), w.h * DH + c * 64, y + r);
                    ++ck;
                    ok = mbar_wait(BAR(C::B_VEMPTY + vs), ((cv / KSTV) & 1u) ^ 1u, abort_flag, wait_ns);
                    if (!ok) break;
                    mbar_expect_tx(BAR(C::B_VFULL + vs), (uint32_t)C::KVBYTES);
#pragma unroll
                    for (int c = 0; c < DH / 64; ++c)
#pragma unroll
                        for (int r = 0; r < BN; r += BOX)
                            tma_load_2d(sV + vs * C::KVBYTES + c * (BN * 128) + r * 128, &tmv, BAR(C::B_VFULL + vs), w.h * DH + c * 64, y + r);
                    ++cv;
                }
            }
            // let every copy this thread issued land before the CTA can exit: the
            // last one of each stage (a stage's earlier phases have been consumed, and
            // a wait for one of them would run into the phase after the last)
            for (uint32_t k = (ck > KSTK ? ck - KSTK : 0); k < ck; ++k) mbar_drain(BAR(C::B_KFULL + k % KSTK), (k / KSTK) & 1u);
            for (uint32_t k = (cv > KSTV ? cv - KSTV : 0); k < cv; ++k) mbar_drain(BAR(C::B_VFULL + k % KSTV), (k / KSTV) & 1u);
        } else if (warp == 1 || warp == 2) {
            // ------------------------------------------------------------------
            // MMA issuer of query tile q (the whole warp walks, one thread issues).
            // Per tile t: S_q(t + 1), then O_q += P_q(t) V(t) (d = 128: the other
            // way round, P_q lies over S_q).  A warp for each tile, because a wait
            // takes 200 to 300 clk beside the softmax warps' exps, even for a
            // barrier that has completed; one warp with both tiles' seven waits
            // took 3 070 clk per tile.
            // ------------------------------------------------------------------
            const uint32_t q = (uint32_t)uniform(warp - 1);
            constexpr uint32_t ID_S = idesc_bf16(BQ, BN, false), ID_PV = idesc_bf16(BQ, DH, true);
            const uint32_t tm = (uint32_t)uniform((int)tmem);
            const uint64_t dq0 = desc_sw128((uint32_t)uniform((int)sQ) + q * C::QBYTES, 16, 1024);
            const uint64_t dk0 = desc_sw128((uint32_t)uniform((int)sK), 16, 1024);
            const uint64_t dv0 = desc_sw128((uint32_t)uniform((int)sV), BN * 128, 1024);
            const uint32_t s_col = tm + C::S_COL + BN * q, p_col = tm + C::P_COL + C::P_STEP * q, o_col = tm + C::O_COL + DH * q;
            constexpr uint32_t STAGE16 = C::KVBYTES >> 4;
            uint32_t ks = 0, kph = 0, vs = 0, vph = 0;     // stage and phase of the next K and V tile
            uint32_t tpar = 0, ipar = 0;                   // score tiles and items so far, mod 2
            bool ok = true;
            const int itb = uniform(it_begin), ite = uniform(it_end);
            const auto next_k = [&] { if (++ks == KSTK) { ks = 0; kph ^= 1u; } };
            const auto next_v = [&] { if (++vs == KSTV) { vs = 0; vph ^= 1u; } };
            // S_q of K stage ks (its operands are there)
            const auto issue_s = [&] {
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t dk = dk0 + ks * STAGE16;
#pragma unroll
                    for (int kk = 0; kk < DH / 16; ++kk) {
                        const uint32_t off = (uint32_t)((kk >> 2) * (BN * 128) + (kk & 3) * 32) >> 4;
                        tc_mma(s_col, dq0 + off, dk + off, ID_S, kk > 0 ? 1u : 0u);
                    }
                    tc_commit(BAR(C::B_SFULL + q));
                    tc_commit(BAR(C::B_KEMPTY + ks));
                }
                __syncwarp();
                next_k();
            };
#define WAIT(bar, parity) mbar_wait_warp(BAR(bar), (parity) & 1u, abort_flag, wait_ns)
            for (int it = itb; it < ite && ok; ++it) {
                const WorkItem w = a.items[it];
                const int n = uniform(w.tile_end - w.tile_begin);
                if (n <= 0) continue;
                if (q == 1u && uniform(__ldg(&a.ranges[w.u].cnt) - w.qt * 2 * BQ) <= BQ) {
                    // no rows in this tile: its K and V tiles pass by
                    for (int t = 0; t < n && ok; ++t) {
                        ok = WAIT(C::B_KFULL + ks, kph);
                        if (!ok) break;
                        if (elect_one()) mbar_arrive(BAR(C::B_KEMPTY + ks));
                        next_k();
                        ok = WAIT(C::B_VFULL + vs, vph);
                        if (!ok) break;
                        if (elect_one()) mbar_arrive(BAR(C::B_VEMPTY + vs));
                        next_v();
                    }
                    continue;
                }
                // S_q(0); at d = 64 it overwrites scores that have to be read
                ok = WAIT(C::B_KFULL + ks, kph) && WAIT(C::B_QFULL + q, ipar) &&
                     (!C::PSEP || WAIT(C::B_SFREE + q, tpar ^ 1u));
                if (!ok) break;
                issue_s();
                for (int t = 0; t < n; ++t) {
                    const uint32_t par = tpar + (uint32_t)t;
                    if (C::PSEP && t + 1 < n) {
                        ok = WAIT(C::B_KFULL + ks, kph) && WAIT(C::B_SFREE + q, par);
                        if (!ok) break;
                        issue_s();
                    }
                    ok = (t > 0 || WAIT(C::B_OFREE + q, ipar ^ 1u)) && WAIT(C::B_VFULL + vs, vph) && WAIT(C::B_PFULL + q, par);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t dv = dv0 + vs * STAGE16;
#pragma unroll
                        for (int kk = 0; kk < BN / 16; ++kk)
                            tc_mma_ts(o_col, p_col + 8u * kk, dv + (uint32_t)((kk * 2048) >> 4), ID_PV, t == 0 && kk == 0 ? 0u : 1u);
                        tc_commit(BAR(C::B_PVDONE + q));
                        tc_commit(BAR(C::B_VEMPTY + vs));
                    }
                    __syncwarp();
                    next_v();
                    if (!C::PSEP && t + 1 < n) {
                        ok = WAIT(C::B_KFULL + ks, kph);
                        if (!ok) break;
                        issue_s();
                    }
                }
                tpar ^= (uint32_t)n & 1u;
                ipar ^= 1u;
            }
#undef WAIT
            // every MMA completes before TMEM is released
            if (elect_one()) {
                tc_commit(BAR(C::B_DRAIN));
                mbar_drain(BAR(C::B_DRAIN), 0);
            }
        }
    } else {
        // ----------------------------------------------------------------------
        // softmax warpgroups: thread = row r of query tile q
        // ----------------------------------------------------------------------
        reg_inc<C::REGS_SOFTMAX>();
        const int q = (warp >> 2) - 1, w4 = warp & 3, r = 32 * w4 + lane;
        const uint32_t tl = tmem + ((uint32_t)(32 * w4) << 16);       // this warp's TMEM lanes
        const uint32_t scol = tl + C::S_COL + (uint32_t)(BN * q), pcol = tl + C::P_COL + C::P_STEP * q;
        const uint32_t ocol = tl + C::O_COL + (uint32_t)(DH * q);
        const float sc = a.scale_log2;
        uint32_t tq = 0;
        int q_loaded = -1;                                             // item whose query rows are in shared memory
        // kept row of item w: its cell, or -1
        auto row_cell = [&](const WorkItem &w, int cnt) {
            const int j = w.qt * 2 * BQ + q * BQ + r;
            if (j >= cnt) return -1;
            const int cell = a.idx[(int64_t)w.u * a.k_max + j];
            return cell < 0 || cell >= a.mn ? 0 : cell;
        };
        auto load_q = [&](const WorkItem &w, int cell) {
            const int g = a.unit_group[w.u];
            const uint16_t *qrow = cell >= 0 ? static_cast<const uint16_t *>(a.q) + ((int64_t)g * a.mn + cell) * a.D + w.h * DH
                                             : nullptr;
            store_q_row<DH>(sQ + q * C::QBYTES, r, qrow, a.rope && cell >= 0 ? a.rope + (int64_t)cell * DH : nullptr);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(BAR(C::B_QFULL + q));
        };
        bool ok = true;
        for (int it = it_begin; it < it_end; ++it) {
            const WorkItem w = a.items[it];
            const RangeSet *rs = a.ranges + w.u;
            const int cnt = __ldg(&rs->cnt), n = w.tile_end - w.tile_begin;
            if (q == 1 && cnt - w.qt * 2 * BQ <= BQ) continue;         // this tile has no rows
            const int cell = row_cell(w, cnt);
            if (n > 0 && q_loaded != it) load_q(w, cell);
            TileWalk walk(rs, w.tile_begin);
            float m_run = -INFINITY, l_run = 0.f;
            for (int j = 0; j < n; ++j) {
                const uint32_t tj = tq + (uint32_t)j;
                const int nv = walk.next();
                ok = mbar_wait_warp(BAR(C::B_SFULL + q), tj & 1u, abort_flag, wait_ns);
                if (!ok) break;
                tc_fence_after();
                uint32_t sr[BN], pk[BN / 2];
                tmem_ld_cols<BN>(scol, sr);
                tmem_wait_ld();
                if (C::PSEP) {                                         // the scores are in registers: S_q may take tile j + 1
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(BAR(C::B_SFREE + q));
                }
                if (nv < BN) mask_cols(sr, nv);
                // The reference moves at the first tile, and when a score passes it by
                // more than 2^8; O (complete up to tile j - 1) and l follow it.
                const float mt = row_max(sr) * sc;
                if (j == 0) {
                    m_run = mt;
                } else if (__any_sync(0xffffffffu, mt > m_run + 8.0f)) {
                    const float m_new = fmaxf(m_run, mt), alpha = ex2_approx(m_run - m_new);
                    ok = mbar_wait_warp(BAR(C::B_PVDONE + q), (tj - 1u) & 1u, abort_flag, wait_ns);
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll 1
                    for (int c = 0; c < DH; c += 16) {
                        uint32_t o[16];
                        tmem_ld16(ocol + (uint32_t)c, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                        tmem_st16(ocol + (uint32_t)c, o);
                    }
                    l_run *= alpha;
                    m_run = m_new;
                }
                const float sum = row_exp(sr, pk, sc, m_run);
                l_run += sum;
                if (C::PSEP && j > 0) {                                // P_q(j - 1) has been read
                    ok = mbar_wait_warp(BAR(C::B_PVDONE + q), (tj - 1u) & 1u, abort_flag, wait_ns);
                    if (!ok) break;
                }
                tc_fence_after();
                tmem_st_cols<BN / 2>(pcol, pk);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(BAR(C::B_PFULL + q));
            }
            if (!ok) break;
            // the next item's query rows, while the last P V runs (every S of this
            // item has been read, so nothing reads the old rows)
            if (n > 0) {
                int nx = it + 1;
                for (; nx < it_end; ++nx) {
                    const WorkItem x = a.items[nx];
                    if (x.tile_end <= x.tile_begin) continue;
                    const int xc = __ldg(&a.ranges[x.u].cnt);
                    if (q == 1 && xc - x.qt * 2 * BQ <= BQ) continue;
                    load_q(x, row_cell(x, xc));
                    q_loaded = nx;
                    break;
                }
                ok = mbar_wait_warp(BAR(C::B_PVDONE + q), (tq + (uint32_t)n - 1u) & 1u, abort_flag, wait_ns);
                if (!ok) break;
                tc_fence_after();
            }
            tq += (uint32_t)n;
            const float inv = l_run > 0.f ? 1.0f / l_run : 0.f;
            const int64_t ooff = ((int64_t)w.u * a.mn + cell) * a.D + w.h * DH;
            float *po = a.part_o + ((int64_t)w.slot * 2 * BQ + q * BQ + r) * DH;
#pragma unroll 1
            for (int c0 = 0; c0 < DH; c0 += 32) {
                uint32_t o[32];
                uint4 res[4];
                if (w.slot < 0 && cell >= 0) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        res[k] = a.residual ? __ldg(reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(a.residual) + ooff + c0) + k)
                                            : make_uint4(0u, 0u, 0u, 0u);
                }
                __syncwarp();                                          // rows without a query took no part above
                if (n > 0) {
                    tmem_ld32(ocol + (uint32_t)c0, o);
                    tmem_wait_ld();
                    if (c0 + 32 == DH) {                               // O_q is read: the next item's P V may start
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(BAR(C::B_OFREE + q));
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) o[e] = 0u;
                }
                if (cell < 0) continue;
                if (w.slot >= 0) {                                     // split-KV partial (fp32, unnormalised)
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        __stcg(reinterpret_cast<float4 *>(po + c0) + k,
                               make_float4(__uint_as_float(o[4 * k]), __uint_as_float(o[4 * k + 1]),
                                           __uint_as_float(o[4 * k + 2]), __uint_as_float(o[4 * k + 3])));
                } else {                                               // out = residual + O / l, rounded once
                    uint4 *dp = reinterpret_cast<uint4 *>(static_cast<uint16_t *>(a.out) + ooff + c0);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t xw[4] = {res[k].x, res[k].y, res[k].z, res[k].w};
                        uint32_t pw[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            pw[e] = pack_bf16x2(__uint_as_float(xw[e] << 16) + __uint_as_float(o[8 * k + 2 * e]) * inv,
                                                __uint_as_float(xw[e] & 0xffff0000u) + __uint_as_float(o[8 * k + 2 * e + 1]) * inv);
                        dp[k] = make_uint4(pw[0], pw[1], pw[2], pw[3]);
                    }
                }
            }
            if (w.slot >= 0 && cell >= 0)
                reinterpret_cast<float2 *>(a.part_ml)[(int64_t)w.slot * 2 * BQ + q * BQ + r] = make_float2(m_run, l_run);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
    if (threadIdx.x == 0 && *abort_flag) latch_status(a.status, RS3_ETIMEOUT);
#undef BAR
}

// The kernel that the plan chose, on the same threads.
template <int DH>
__global__ void __launch_bounds__(NTHREADS, 1)
k_readout_either(const ReadoutArgs a, const __grid_constant__ CUtensorMap tmk, const __grid_constant__ CUtensorMap tmv)
{
    static_assert(NTHREADS == tc::Cfg<DH>::NTHREADS, "one launch for both");
    // set up for the one-tile kernel, whose calls are the short ones
    const uint32_t tmem = set_up_tc<DH>(tmk, tmv);
    pdl_wait();                      // the plan
    const int first = a.cta_items[2 * blockIdx.x], it_end = a.cta_items[2 * blockIdx.x + 1];
    if (first & RS3_PAIR_ITEMS) readout_pair<DH>(a, tmk, tmv, tmem, first & ~RS3_PAIR_ITEMS, it_end);
    else readout_tc<DH>(a, tmk, tmv, tmem, first, it_end);
}

template <int DH>
rs3_status launch(const ReadoutArgs &a, cudaStream_t st)
{
    constexpr int smem = Cfg<DH>::SMEM > tc::Cfg<DH>::SMEM ? Cfg<DH>::SMEM : tc::Cfg<DH>::SMEM;
    if (rs3_kernel_smem((const void *)k_readout_either<DH>, smem) != RS3_OK) return RS3_ECUDA;
    const int64_t rows = (int64_t)a.U * a.rows_per_unit;
    if (rows >= (int64_t)1 << 31) return RS3_EUNSUPPORTED;
    CUtensorMap mk, mv;
    if (!make_kv_map(&mk, a.k_store, a.D, rows, tc::Cfg<DH>::BN) || !make_kv_map(&mv, a.v_store, a.D, rows, tc::Cfg<DH>::BN))
        return RS3_ECUDA;
    launch_pdl(k_readout_either<DH>, dim3((unsigned)a.grid_ctas), dim3(NTHREADS), smem, st, a, mk, mv);
    return cudaGetLastError() == cudaSuccess ? RS3_OK : RS3_ECUDA;
}

}  // namespace pair

}  // namespace tc

rs3_status rs3_launch_either_readout(const ReadoutArgs &a, cudaStream_t st)
{
    switch (a.d) {
    case 64: return tc::pair::launch<64>(a, st);
    case 128: return tc::pair::launch<128>(a, st);
    default: return RS3_EUNSUPPORTED;
    }
}
