// rs3_readout_tc.cu -- the one-tile tensor-core readout (rs3_readout_tc.cuh) as a
// kernel of its own: heads of 256, and calls that the two-tile kernel has no part in.
#include "rs3_readout_tc.cuh"

namespace tc {

template <int DH>
__global__ void __launch_bounds__(Cfg<DH>::NTHREADS, 1)
k_readout_tc(const ReadoutArgs a, const __grid_constant__ CUtensorMap tmk, const __grid_constant__ CUtensorMap tmv)
{
    const uint32_t tmem = set_up_tc<DH>(tmk, tmv);
    pdl_wait();                      // the plan
    readout_tc<DH>(a, tmk, tmv, tmem, a.cta_items[2 * blockIdx.x], a.cta_items[2 * blockIdx.x + 1]);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <int DH>
rs3_status launch(const ReadoutArgs &a, cudaStream_t st)
{
    if (rs3_kernel_smem((const void *)k_readout_tc<DH>, Cfg<DH>::SMEM) != RS3_OK) return RS3_ECUDA;
    const int64_t rows = (int64_t)a.U * a.rows_per_unit;
    if (rows >= (int64_t)1 << 31) return RS3_EUNSUPPORTED;
    CUtensorMap mk, mv;
    if (!make_kv_map(&mk, a.k_store, a.D, rows, Cfg<DH>::BN) ||
        !make_kv_map(&mv, a.v_store, a.D, rows, Cfg<DH>::BN))
        return RS3_ECUDA;
    const int64_t grid = a.grid_ctas;               // the plan's slices; unused ones exit at once
    launch_pdl(k_readout_tc<DH>, dim3((unsigned)grid), dim3(Cfg<DH>::NTHREADS), Cfg<DH>::SMEM, st, a, mk, mv);
    return cudaGetLastError() == cudaSuccess ? RS3_OK : RS3_ECUDA;
}

}  // namespace tc

bool rs3_tc_supported(int d) { return d == 64 || d == 128 || d == 256; }

int rs3_tc_block_n(int d)
{
    switch (d) {
    case 64: return tc::Cfg<64>::BN;
    case 128: return tc::Cfg<128>::BN;
    default: return tc::Cfg<256>::BN;
    }
}

rs3_status rs3_launch_tc_readout(const ReadoutArgs &a, cudaStream_t st)
{
    switch (a.d) {
    case 64: return tc::launch<64>(a, st);
    case 128: return tc::launch<128>(a, st);
    case 256: return tc::launch<256>(a, st);
    default: return RS3_EUNSUPPORTED;
    }
}
