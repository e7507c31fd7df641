// pd_force_lps.cu -- state-based linear peridynamic solid (LPS): the dilatation
// pass and the force pass of Algorithm 2, the latter fused with the explicit
// update (Eq. (4); Eqs. (7)-(9)).
//
// In lattice units (xi = d, e~ = e / h, m~ = m / (h^2 V), omega = 1):
//   e~      = (2 d.eta + eta.eta) / (|y| + |d|)          cancellation-free extension
//   theta_i = (3 / m~_i) sum_j |d| e~ V_ij                Algorithm 2, second loop
//   f_i     = (1/h) sum_j [ (3K - 5mu) |d| (a_i + a_j) + 15 mu e~ (b_i + b_j) ] V_ij y/|y|
// with a = theta / m~, b = 1 / m~. The bracket is t_i<xi> + t_j<-xi> of Algorithm
// 2's third loop (t = 3K theta |xi| / m + 15 mu e^d / m, e^d = e - theta |xi| / 3)
// gathered at i: the "f_j -= t M V_i" scatter of row j lands on i as + t_j M_ij.
// The weighted volume m~ is computed once at the neighbour build.
#include <string.h>

#include "pd_lps_fast.cuh"

namespace pdk {

int launch_rows_lps(const TileArgs &a, const RowArgs &ra, int dil, cudaStream_t st);
size_t rows_smem(const RowArgs &ra, bool force, bool param_table);
int launch_f64_lps(const TileArgs &a, int dil, size_t smem, cudaStream_t st);

size_t lps_fast_smem(const Geom &g, bool dil)
{
    const size_t n = (size_t)(g.bx + 2 * g.m) * (g.by + 2 * g.m) * (g.bz / 2 + 2 * g.m);
    const size_t p2 = ((n + 1) / 2) * sizeof(float4);
    if (dil) return n * sizeof(float4) + p2 + (size_t)g.S * 3 * sizeof(float4);
    return 2 * n * sizeof(float4) + p2 + (size_t)g.S * 3 * sizeof(float4);
}

// ---------------------------------------------------------------- dispatch

size_t lps_generic_smem(const Geom &g, int precision, bool dil)
{
    if (precision != PD_FP64) return lps_fast_smem(g, dil);
    const size_t nbox = (size_t)(g.bx + 2 * g.m) * (g.by + 2 * g.m) * (g.bz + 2 * g.m);
    return nbox * (sizeof(double4_32a) + (dil ? 0 : sizeof(double)));
}

// dil = 1: dilatation pass; dil = 0: force pass (+ update per a.mode).
int launch_lps_args(const TileArgs &a, int precision, int dil, cudaStream_t st)
{
    const Geom &g = a.g;
    const size_t smem = lps_generic_smem(g, precision, dil);
    if (precision == PD_FP32C && a.rows && (dil ? rows_dil(g) : rows_frc(g, rows_smem(a.rows[1], true, false))))
        return launch_rows_lps(a, a.rows[dil ? 0 : 1], dil, st);
    if (precision == PD_FP32C) {
        // dilatation: two pairs per thread from 2^7-point tiles and two stencil words on
        const bool dil2 = dil && g.T >= 128 && g.W >= 2;
        const int threads = dil ? (g.T / 2 < 256 ? g.T / 2 : 256) : g.T;
        static thread_local ParamTab tp;
        // the table as a kernel parameter on grids of several waves (as for PMB,
        // pd_force_pmb.cu): 128^3 force pass 0.392 -> 0.361 ms
        // (the dilatation's table is tab_a, the force pass's tab_b)
        const float4 *ht = dil ? a.htab_a : a.htab_b;
        const int nt = dil ? a.ntab_a : a.ntab_b;
        const bool pt = ht && nt > 0 && nt <= PTAB_N && g.ntiles >= PTAB_MIN_TILES;
        if (pt) {
            memcpy(tp.e, ht, sizeof(float4) * (size_t)nt);
            auto k = dil ? (dil2 ? (a.vol_corr ? lps_dil_fast2_pt<true> : lps_dil_fast2_pt<false>)
                                 : (a.vol_corr ? lps_dil_fast_pt<true> : lps_dil_fast_pt<false>))
                         : (a.vol_corr ? lps_force_fast_pt<true> : lps_force_fast_pt<false>);
            PD_CUDA(smem_limit(k, smem));
            k<<<g.ntiles, threads, smem, st>>>(a, tp);
        } else {
            const bool cols = cols_staging(a) && (g.ntiles >= ROWS_MIN_TILES || ragged(a));
            auto k = dil ? (dil2 ? (cols ? (a.vol_corr ? lps_dil_fast2<true, true> : lps_dil_fast2<false, true>)
                                         : (a.vol_corr ? lps_dil_fast2<true, false> : lps_dil_fast2<false, false>))
                                 : (a.vol_corr ? lps_dil_fast<true> : lps_dil_fast<false>))
                         : (a.vol_corr ? lps_force_fast<true> : lps_force_fast<false>);
            PD_CUDA(smem_limit(k, smem));
            k<<<g.ntiles, threads, smem, st>>>(a);
        }
    } else {
        return launch_f64_lps(a, dil, smem, st);
    }
    PD_CUDA(cudaGetLastError());
    return PD_OK;
}

}  // namespace pdk
