// pd_rows.cu -- kernels and launches of the row-wise FP32C passes (pd_rows.cuh).
#include "pd_rows.cuh"

namespace pdk {

// CTAs per SM the kernels are built for: 64 registers for four (three at 80 registers:
// 128^3 PMB step 0.247 -> 0.256 ms, dilatation 0.190 -> 0.200 ms); the LPS force pass 80 for
// three on grids of several waves (0.327 -> 0.320 ms against two), 128 for two below
// (64^3: 0.066 -> 0.059 ms against three).
template <int LAW, bool PT>
constexpr int rows_ctas()
{
    return LAW == ROW_FRC ? (PT ? 3 : 2) : 4;
}

template <int LAW, bool VOL, int PARTS>
__global__ void __launch_bounds__(256, rows_ctas<LAW, false>())
    rows(const __grid_constant__ TileArgs a, const __grid_constant__ RowArgs ra)
{
    rows_body<LAW, VOL, PARTS, false>(a, ra, blockIdx.x, nullptr);
}

template <int LAW, bool VOL, int PARTS>
__global__ void __launch_bounds__(256, rows_ctas<LAW, true>())
    rows_pt(const __grid_constant__ TileArgs a, const __grid_constant__ RowArgs ra, const __grid_constant__ RowTab tab)
{
    rows_body<LAW, VOL, PARTS, true>(a, ra, blockIdx.x, tab.e);
}

size_t rows_smem(const RowArgs &ra, bool force, bool param_table)
{
    const size_t n = ra.nbox;
    return (n * (force ? 2 : 1) + (n + 1) / 2 + (param_table ? 0 : ra.ntab)) * sizeof(float4);
}

template <int LAW, bool VOL, int PARTS>
static int go_parts(const TileArgs &a, const RowArgs &ra, cudaStream_t st)
{
    // the table as a kernel parameter on grids of several waves, as for the word-wise
    // kernels (pd_force_pmb.cu)
    const bool pt = ra.ntab <= ROWS_PTAB && a.g.ntiles >= PTAB_MIN_TILES;
    const size_t smem = rows_smem(ra, LAW == ROW_FRC, pt);
    if (pt) {
        static thread_local RowTab tab;
        memcpy(tab.e, ra.htab, sizeof(float4) * (size_t)ra.ntab);
        PD_CUDA(smem_limit(rows_pt<LAW, VOL, PARTS>, smem));
        rows_pt<LAW, VOL, PARTS><<<a.g.ntiles, 256, smem, st>>>(a, ra, tab);
    } else {
        PD_CUDA(smem_limit(rows<LAW, VOL, PARTS>, smem));
        rows<LAW, VOL, PARTS><<<a.g.ntiles, 256, smem, st>>>(a, ra);
    }
    PD_CUDA(cudaGetLastError());
    return PD_OK;
}

template <int LAW, bool VOL>
static int go(const TileArgs &a, const RowArgs &ra, cudaStream_t st)
{
    return ra.parts == 2 ? go_parts<LAW, VOL, 2>(a, ra, st) : go_parts<LAW, VOL, 1>(a, ra, st);
}

int launch_rows_pmb(const TileArgs &a, const RowArgs &ra, cudaStream_t st) { return go<ROW_PMB, false>(a, ra, st); }

int launch_rows_lps(const TileArgs &a, const RowArgs &ra, int dil, cudaStream_t st)
{
    if (dil) return a.vol_corr ? go<ROW_DIL, true>(a, ra, st) : go<ROW_DIL, false>(a, ra, st);
    return a.vol_corr ? go<ROW_FRC, true>(a, ra, st) : go<ROW_FRC, false>(a, ra, st);
}

}  // namespace pdk
