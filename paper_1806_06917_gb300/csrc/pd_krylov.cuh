// pd_krylov.cuh -- what the two forms of the Krylov solvers share: a kernel per operation
// (pd_krylov.cu) and a GMRES cycle in one cooperative launch (pd_krylov_grid.cu).
#pragma once

#include <math.h>

#include <algorithm>

#include "pd_tile.cuh"

namespace pdk {

constexpr int KT = 256;               // threads per block
constexpr int KPER = 8;               // elements per thread in a reduction block
constexpr int KCHUNK = KT * KPER;     // elements per reduction block

__host__ __device__ inline int kblocks(long long n) { return (int)((n + KCHUNK - 1) / KCHUNK); }

// Fixed-order sum of one value per thread of the block; the result is valid in
// thread 0.
__device__ __forceinline__ double block_sum(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    __syncthreads();            // red may still be read from a previous call
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < KT / 32; ++w) t += red[w];
    return t;
}

// Device layout of GMRES's small arrays in dsc (m = restart): the dot results
// [0, m+1), the Hessenberg matrix H (column-major, (m+1) x m), the rotations cs
// and sn, the rotated right-hand side g (m+1), the solution y of the small
// triangular system (m), and the scalars. The host reads the scalars back once
// per chunk of Arnoldi steps (a kernel per operation) or once per cycle (one
// launch); a step after the one that met the target (or broke down) changes
// nothing that the update of x uses.
struct GmLayout {
    int m, H, cs, sn, g, y, sc;
    __host__ __device__ explicit GmLayout(int m_)
        : m(m_), H(m_ + 1), cs(H + (m_ + 1) * m_), sn(cs + m_), g(sn + m_), y(g + m_ + 1), sc(y + m_)
    {
    }
    __host__ __device__ int size() const { return sc + 8; }
};
enum { GM_TARGET = 0, GM_DONE, GM_K, GM_RES, GM_INVH, GM_ITERS };

// After |w|^2 = ww: H[j+1, j] = |w|, the previous rotations and a new one on column j, g
// rotated, the residual estimate |g[j+1]|, the scale 1/|w| for w; nothing once the cycle
// is done. The block stages column j and the rotations in shared memory gs (3 (m + 1)
// doubles) so that the sequential rotation loop of thread 0 does not wait on global loads.
__device__ __forceinline__ void gm_givens(double *d, int m, int j, double ww, double *gs)
{
    const GmLayout L(m);
    double *sc = d + L.sc;
    if (sc[GM_DONE] != 0.0) {
        if (threadIdx.x == 0) sc[GM_INVH] = 0.0;
        return;
    }
    double *hj = d + L.H + (m + 1) * j;
    double *hs = gs, *css = gs + (m + 1), *sns = gs + 2 * (m + 1);
    for (int i = threadIdx.x; i <= j; i += blockDim.x) hs[i] = hj[i];
    for (int i = threadIdx.x; i < j; i += blockDim.x) {
        css[i] = d[L.cs + i];
        sns[i] = d[L.sn + i];
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double hn = sqrt(ww);
    double *cs = d + L.cs, *sn = d + L.sn, *g = d + L.g;
    hs[j + 1] = hn;
    for (int i = 0; i < j; ++i) {
        const double t = css[i] * hs[i] + sns[i] * hs[i + 1];
        hs[i + 1] = -sns[i] * hs[i] + css[i] * hs[i + 1];
        hs[i] = t;
    }
    const double den = hypot(hs[j], hs[j + 1]);
    cs[j] = den > 0.0 ? hs[j] / den : 1.0;
    sn[j] = den > 0.0 ? hs[j + 1] / den : 0.0;
    hs[j] = den;
    hs[j + 1] = 0.0;
    for (int i = 0; i <= j + 1; ++i) hj[i] = hs[i];
    g[j + 1] = -sn[j] * g[j];
    g[j] = cs[j] * g[j];
    sc[GM_K] = j + 1;
    sc[GM_ITERS] += 1.0;
    sc[GM_RES] = fabs(g[j + 1]);
    sc[GM_INVH] = hn > 0.0 ? 1.0 / hn : 0.0;
    if (sc[GM_RES] <= sc[GM_TARGET] || hn == 0.0) sc[GM_DONE] = 1.0;
}

// Blocks of the grid form at most (one per SM).
constexpr int GRID_MAX = 256;

// The grid form: steps 0 .. steps - 1 of a GMRES cycle from V_0 and the scalars in d, whose
// last double (after GmLayout's) is the barrier. PD_ENOTREADY where the launch is not possible
// (nothing has run).
int gmres_grid(const TanOp &t, double *V, long long n, double *partial, double *d, int m, int steps, long long wait_ns,
               int stall, cudaStream_t st);

}  // namespace pdk
