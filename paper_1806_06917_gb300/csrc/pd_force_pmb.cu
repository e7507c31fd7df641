// pd_force_pmb.cu -- bond-based PMB internal force with bond breaking, fused
// with the explicit update (Eq. (3); Algorithm 1's loop over points and their
// horizons; Eqs. (7)-(9) for the update).
//
// Per bond, in lattice units (xi = d, integer; eta = u~_j - u~_i):
//   y   = d + eta,   q = |y|^2,   r = |y| = q rsqrt(q)
//   s   = (2 d.eta + eta.eta) / (|d| (r + |d|))      cancellation-free stretch
//   f_i += c V V_ij s y / r                          (PMB pair force)
// A bond breaks for good when s > s_c, tested before it contributes. Each point
// sums its bonds sequentially in stencil order: no atomics, deterministic.
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "pd_pmb_fast.cuh"

// Unroll depth of np_fast's bond loops.
#ifndef PD_NP_UNROLL
#define PD_NP_UNROLL PD_UNROLL
#endif
// Bonds of a row unrolled in np_rows (443^2, m = 20: 0.1338 ms with 4, 0.1323 with 8, 0.1325
// with 12).
#ifndef PD_NP_ROW
#define PD_NP_ROW 8
#endif

namespace pdk {

int launch_rows_pmb(const TileArgs &a, const RowArgs &ra, cudaStream_t st);
int launch_f64_bonds(const TileArgs &a, size_t smem, cudaStream_t st);

// Paired halo box (float4 {x_A, x_B, y_A, y_B}, plus float2 {z_A, z_B} in 3D)
// followed by the stencil table of `words` float4 per entry.
static size_t fast_smem(const Geom &g, int words)
{
    size_t n;
    if (g.dim == 3) n = (size_t)(g.bx + 2 * g.m) * (g.by + 2 * g.m) * (g.bz / 2 + 2 * g.m);
    else n = (size_t)(g.bx + 2 * g.m) * (g.by / 2 + 2 * g.m);
    const size_t p2 = g.dim == 3 ? ((n + 1) / 2) * sizeof(float4) : 0;
    return n * sizeof(float4) + p2 + (size_t)g.S * words * sizeof(float4);
}

size_t pmb_fast_smem(const Geom &g) { return fast_smem(g, 4); }

size_t np_fast_smem(const Geom &g) { return fast_smem(g, NP_TAB_WORDS(g.dim)); }

// ------------------------------------------------------------- NP / LP, FP32C

// One 32-bond word of the NP / LP sum (Algorithm 1) for a point pair in f32x2.
// With S = eta.d / |d|^2 the bond term is t S [exp2(a S^2) for NP] d, t = J
// V_ij / |d| and a = -beta h |d| / ln 2 (see pd_api.cu); written in p = eta.d:
//   w = k p [exp2(a' p^2) for NP],  F += w d,   k = t / |d|^2,  a' = a / |d|^4.
// The direction is the reference bond d, so no square root or reciprocal is
// needed. Table entries of NP_TAB_WORDS(DIM) float4, the fewest shared-memory
// wavefronts per bond (a broadcast 16-byte load costs two):
//   2D: {dx,dx,dy,dy} {k,k,a',offset}
//   3D: {dx,dx,dy,dy} {dz,dz,k,k} {a',offset,-,-}
template <int DIM, bool MASKED, bool LINEAR>
__device__ __forceinline__ void np_word(const float4 *tw, int nb, const float4 *P4, const float2 *P2, int bi,
                                        float2 nux, float2 nuy, float2 nuz, uint32_t c0, uint32_t c1, float2 &Fx,
                                        float2 &Fy, float2 &Fz)
{
    constexpr int E = NP_TAB_WORDS(DIM);
PD_PRAGMA_UNROLL(PD_NP_UNROLL)
    for (int b = 0; b < nb; ++b) {
        const float4 ta = tw[E * b], tb = tw[E * b + 1];
        float ak;
        int off;
        if (DIM == 3) {
            const float2 tc = reinterpret_cast<const float2 *>(tw + E * b + 2)[0];
            ak = tc.x;
            off = __float_as_int(tc.y);
        } else {
            ak = tb.z;
            off = __float_as_int(tb.w);
        }
        const float4 r4 = P4[bi + off];
        const float2 ex = f2add(f2lo(r4), nux), ey = f2add(f2hi(r4), nuy);
        float2 dot = f2mul(ex, f2lo(ta));
        dot = f2fma(ey, f2hi(ta), dot);
        if (DIM == 3) dot = f2fma(f2add(P2[bi + off], nuz), f2lo(tb), dot);
        float2 wgt = f2mul(dot, DIM == 3 ? f2hi(tb) : f2lo(tb));
        if (!LINEAR) wgt = f2mul(wgt, f2ex2(f2mul(make_float2(ak, ak), f2mul(dot, dot))));
        if (MASKED) {
            wgt.x = ((c0 >> b) & 1u) ? wgt.x : 0.f;
            wgt.y = ((c1 >> b) & 1u) ? wgt.y : 0.f;
        }
        Fx = f2fma(wgt, f2lo(ta), Fx);
        Fy = f2fma(wgt, f2hi(ta), Fy);
        if (DIM == 3) Fz = f2fma(wgt, f2lo(tb), Fz);
    }
}

template <int DIM, bool LINEAR, bool SPLIT>
__global__ void __launch_bounds__(SPLIT ? 1024 : 256, SPLIT ? 1 : PD_MINBLOCKS) np_fast(const TileArgs a)
{
    const Geom &g = a.g;
    const PairBox pb = pair_box(g);
    const int S = g.S;
    extern __shared__ float4 smem4[];
    float4 *P4 = smem4;
    float2 *P2 = reinterpret_cast<float2 *>(P4 + pb.n);
    float4 *tab = P4 + pb.n + (DIM == 3 ? (pb.n + 1) / 2 : 0);      // the layout of np_fast_smem
    constexpr int E = NP_TAB_WORDS(DIM);
    __shared__ int s_nbr[27];
    const int tile = blockIdx.x;
    const int4 org = __ldg(&a.tile_org[tile]);
    for (int k = threadIdx.x; k < E * S; k += blockDim.x) tab[k] = __ldg(&a.tab_a[k]);
    load_nbr(a, tile, s_nbr);
    __syncthreads();
    stage_pairs(a, pb, org, tile, s_nbr, P4, DIM == 3 ? P2 : nullptr, true);
    __syncthreads();

    const int nthr = g.T / 2;            // point pairs; thread (t, part) as in pmb_fast
    const int part = SPLIT ? threadIdx.x / nthr : 0;
    const int w0 = SPLIT ? part * g.W / a.split : 0, w1 = SPLIT ? (part + 1) * g.W / a.split : g.W;
    // one iteration per thread (T / 2 <= 256 = blockDim without the split)
    for (int t = SPLIT ? threadIdx.x % nthr : threadIdx.x; t < nthr; t += SPLIT ? nthr : blockDim.x) {
        const PairPts q = pair_points(g, pb, org, tile, t);
        const float4 ui4 = P4[q.bi];
        const float2 nux = f2neg(f2lo(ui4)), nuy = f2neg(f2hi(ui4));
        const float2 nuz = DIM == 3 ? f2neg(P2[q.bi]) : make_float2(0.f, 0.f);
        float2 Fx = make_float2(0.f, 0.f), Fy = Fx, Fz = Fx;
        const size_t mo0 = (size_t)w0 * g.nslots;
        uint32_t n0 = q.act[0] && (!SPLIT || w0 < w1) ? a.mask[mo0 + q.slot[0]] : 0u;
        uint32_t n1 = q.act[1] && (!SPLIT || w0 < w1) ? a.mask[mo0 + q.slot[1]] : 0u;
        for (int w = w0; w < w1; ++w) {
            const uint32_t m0 = n0, m1 = n1;
            if (w + 1 < w1) {
                const size_t mo = (size_t)(w + 1) * g.nslots;
                n0 = q.act[0] ? a.mask[mo + q.slot[0]] : 0u;
                n1 = q.act[1] ? a.mask[mo + q.slot[1]] : 0u;
            }
            const int nb = min(32, S - 32 * w);
            const uint32_t full = nb == 32 ? 0xffffffffu : ((1u << nb) - 1u);
            const float4 *tw = tab + E * 32 * w;
            if (__all_sync(0xffffffffu, m0 == full && m1 == full))
                np_word<DIM, false, LINEAR>(tw, nb, P4, P2, q.bi, nux, nuy, nuz, m0, m1, Fx, Fy, Fz);
            else
                np_word<DIM, true, LINEAR>(tw, nb, P4, P2, q.bi, nux, nuy, nuz, m0, m1, Fx, Fy, Fz);
        }
        if (SPLIT) pair_split_sum(a, reinterpret_cast<float2 *>(tab + E * S), nthr, t, part, Fx, Fy, Fz);
        if (part == 0) {
            const float FA[3] = {Fx.x, Fy.x, Fz.x}, FB[3] = {Fx.y, Fy.y, Fz.y};
            pair_epilogue2(a, q, FA, FB, DIM);
        }
    }
}

// 2D wide horizons: each thread owns two point pairs adjacent in x, and walks each row of
// the stencil with the box column of its second pair at one bond kept as that of its first
// at the next: a bond of four points takes one gather and the entry's dx, k and a' (dy is
// the row's), 8 shared-memory wavefronts a 32-lane step against 12 with two pairs T / 4
// apart in y. The box is stored as its even columns and then its odd ones, so that a
// gather's lanes are 16 bytes apart and the columns of a row come from the two halves in
// turn at constant offsets. What bounds it: the packed FP32 pipe, 40 cycles a step and
// sub-partition (50,000 cycles of a tile's 68,000 in its bonds, alone on its SM, at m = 20);
// around the bonds, 8,000 cycles for masks and addresses, 9,000 of staging (19,000 with each
// point staged by both of its pairs from a Morton order read row by row and a table of tiles
// in global memory) and 7,000 of update (12,000 by a quarter of the threads), which a younger
// CTA hardly gets on with while an older one has bonds. 443^2, m = 20 (392 tiles on 304
// slots): 0.143 -> 0.132 ms a step. The arithmetic is np_word's, bond by bond.
//
// Bonds [k, kend) of the stencil, which one word holds if MASKED (c0..c3: its masks of the
// four points, from bit 0). A row ends at the disk's edge or before the point itself.
template <bool MASKED, bool LINEAR>
__device__ __forceinline__ void np_row_bonds(const float4 *tab, int m, int k, int kend, const float4 *P4, int half, int bi,
                                             float2 nux0, float2 nuy0, float2 nux1, float2 nuy1, uint32_t c0,
                                             uint32_t c1, uint32_t c2, uint32_t c3, float2 &Fx0, float2 &Fy0,
                                             float2 &Fx1, float2 &Fy1)
{
    while (k < kend) {
        const float4 *tw = tab + 2 * k;
        const float4 first = tw[0];
        const float2 dy = f2hi(first);
        const int dx = (int)first.x, y = (int)first.z;
        const int end = y == 0 && dx < 0 ? -1 : (int)__fsqrt_rn((float)(m * m - y * y));
        int len = min(end - dx + 1, kend - k);
        const int b0 = bi + __float_as_int(tw[1].w), odd = b0 & 1;
        const float4 *A = P4 + (b0 >> 1) + (odd ? half : 0), *B = P4 + (b0 >> 1) + (odd ? 1 : half);
        uint32_t m0 = 0, m1 = 0, m2 = 0, m3 = 0;
        if (MASKED) {
            const int sh = k & 31;
            m0 = c0 >> sh, m1 = c1 >> sh, m2 = c2 >> sh, m3 = c3 >> sh;
        }
        k += len;
        auto bond = [&](const float4 &r0, const float4 &r1, int b) {
            const float2 dxx = reinterpret_cast<const float2 *>(tw + 2 * b)[0];
            const float4 tb = tw[2 * b + 1];
            const float2 ex0 = f2add(f2lo(r0), nux0), ey0 = f2add(f2hi(r0), nuy0);
            const float2 ex1 = f2add(f2lo(r1), nux1), ey1 = f2add(f2hi(r1), nuy1);
            float2 dot0 = f2mul(ex0, dxx), dot1 = f2mul(ex1, dxx);
            dot0 = f2fma(ey0, dy, dot0);
            dot1 = f2fma(ey1, dy, dot1);
            float2 w0 = f2mul(dot0, f2lo(tb)), w1 = f2mul(dot1, f2lo(tb));
            if (!LINEAR) {
                const float2 ak = make_float2(tb.z, tb.z);
                w0 = f2mul(w0, f2ex2(f2mul(ak, f2mul(dot0, dot0))));
                w1 = f2mul(w1, f2ex2(f2mul(ak, f2mul(dot1, dot1))));
            }
            if (MASKED) {
                w0.x = ((m0 >> b) & 1u) ? w0.x : 0.f;
                w0.y = ((m1 >> b) & 1u) ? w0.y : 0.f;
                w1.x = ((m2 >> b) & 1u) ? w1.x : 0.f;
                w1.y = ((m3 >> b) & 1u) ? w1.y : 0.f;
            }
            Fx0 = f2fma(w0, dxx, Fx0);
            Fy0 = f2fma(w0, dy, Fy0);
            Fx1 = f2fma(w1, dxx, Fx1);
            Fy1 = f2fma(w1, dy, Fy1);
        };
        float4 r = A[0];
        auto run = [&](auto n) {       // n bonds (even)
            constexpr int N = decltype(n)::value;
#pragma unroll
            for (int q = 0; q < N / 2; ++q) {
                const float4 rb = B[q], ra = A[q + 1];
                bond(r, rb, 2 * q);
                bond(rb, ra, 2 * q + 1);
                r = ra;
            }
            A += N / 2, B += N / 2, tw += 2 * N;
            if (MASKED) m0 >>= N, m1 >>= N, m2 >>= N, m3 >>= N;
        };
#pragma unroll 1
        for (; len >= PD_NP_ROW; len -= PD_NP_ROW) run(std::integral_constant<int, PD_NP_ROW>());
#pragma unroll 1
        for (; len >= 2; len -= 2) run(std::integral_constant<int, 2>());
        if (len) bond(r, B[0], 0);
    }
}

// Tiles a 2D tile's box reaches, in x and y, to either side.
static __host__ __device__ inline int2 tile_reach(const Geom &g)
{
    return make_int2((g.m + g.bx - 1) >> g.lbx, (g.m + g.by - 1) >> g.lby);
}
constexpr int NP_LUT = 64;

// Launch: one CTA per tile, (tile points / 4) * a.split threads; thread (t, sub) owns pairs
// 2 t and 2 t + 1 and the sub-th of a.split ranges of stencil words.
template <bool LINEAR>
__global__ void __launch_bounds__(1024, 1) np_rows(const TileArgs a)
{
    const Geom &g = a.g;
    const PairBox pb = pair_box(g);
    const int S = g.S, half = pb.n / 2;       // HX = bx + 2 m is even
    extern __shared__ float4 smem4[];
    float4 *P4 = smem4;
    float4 *tab = P4 + pb.n;                  // the layout of np_fast_smem in 2D
    constexpr int E = NP_TAB_WORDS(2);
    __shared__ int s_lut[NP_LUT];
    const int tile = blockIdx.x;
    const int4 org = __ldg(&a.tile_org[tile]);
    for (int k = threadIdx.x; k < E * S; k += blockDim.x)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(&tab[k])), "l"(&a.tab_a[k])
                     : "memory");
    const int2 reach = tile_reach(g);
    const int ncx = 2 * reach.x + 1;
    for (int k = threadIdx.x; k < ncx * (2 * reach.y + 1); k += blockDim.x) {
        const int tx = (org.x >> g.lbx) - reach.x + k % ncx, ty = (org.y >> g.lby) - reach.y + k / ncx;
        const bool in = tx >= 0 && ty >= 0 && (tx << g.lbx) < g.nx && (ty << g.lby) < g.ny;
        s_lut[k] = in ? __ldg(&a.tile_lut[tx + g.tgx * ty]) : -1;
    }
    const int npairs = g.T / 2, nthr = npairs / 2;     // nthr: a multiple of 32 (T >= 128)
    const int sub = threadIdx.x / nthr, t = threadIdx.x % nthr;
    const int w0 = sub * g.W / a.split, w1 = (sub + 1) * g.W / a.split;
    const PairPts q0 = pair_points(g, pb, org, tile, 2 * t), q1 = pair_points(g, pb, org, tile, 2 * t + 1);
    // the words of the points x and x + 1 of a row stand side by side (nslots is even)
    auto word = [&](int w, uint32_t *c) {
        const size_t mo = (size_t)w * g.nslots;
        const uint2 A = *reinterpret_cast<const uint2 *>(&a.mask[mo + q0.slot[0]]);
        const uint2 B = *reinterpret_cast<const uint2 *>(&a.mask[mo + q0.slot[1]]);
        c[0] = q0.act[0] ? A.x : 0u;
        c[1] = q0.act[1] ? B.x : 0u;
        c[2] = q1.act[0] ? A.y : 0u;
        c[3] = q1.act[1] ? B.y : 0u;
    };
    auto full_word = [&](int w) { return S - 32 * w >= 32 ? 0xffffffffu : (1u << (S - 32 * w)) - 1u; };
    // whether the warp has every bond of its range (read beside the staging's loads)
    bool all = true;
#pragma unroll 5
    for (int w = w0; w < w1; ++w) {
        uint32_t c[4];
        word(w, c);
        all = all && (c[0] & c[1] & c[2] & c[3]) == full_word(w);
    }
    all = __all_sync(0xffffffffu, all);
    __syncthreads();
    // Staging: every point of the box once (in a pair of rows each is both an A and a B),
    // two rows side by side, so that a warp's loads share lines of the Morton order; the
    // tiles from the table above (m may span several).
    {
        const Ref32 ref = tile_ref32(a, tile);
        const float inv_h = (float)a.inv_h, inv_row = __frcp_rn((float)(2 * pb.HX));
        const int hb = g.by / 2;
        float *P = reinterpret_cast<float *>(P4);
#pragma unroll 4
        for (int p = threadIdx.x; p < pb.HX * (pb.HY + hb); p += blockDim.x) {
            const int r = fdiv_small(p, inv_row), rem = p - r * 2 * pb.HX, x = rem >> 1, y = 2 * r + (rem & 1);
            const int gx = org.x - g.m + x, gy = org.y - g.m + y;
            int s = -1;
            if ((unsigned)gx < (unsigned)g.nx && (unsigned)gy < (unsigned)g.ny) {
                const int tx = (gx >> g.lbx) - (org.x >> g.lbx) + reach.x, ty = (gy >> g.lby) - (org.y >> g.lby) + reach.y;
                s = s_lut[tx + ncx * ty] * g.T + brick_code(2, gx & (g.bx - 1), gy & (g.by - 1), 0);
            }
            const float4 v = stage_one(a, a.src_hl, s, ref, inv_h);
            float *e = P + 4 * ((y * pb.HX + x) / 2 + (x & 1 ? half : 0));
            if (y < pb.HY) e[0] = v.x, e[2] = v.y;
            if (y >= hb) e -= 2 * hb * pb.HX, e[1] = v.x, e[3] = v.y;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    float2 Fx0, Fy0, Fx1, Fy1;
    Fx0 = Fy0 = Fx1 = Fy1 = make_float2(0.f, 0.f);
    {
        const float4 u0 = P4[(q0.bi >> 1) + (q0.bi & 1 ? half : 0)], u1 = P4[(q1.bi >> 1) + (q1.bi & 1 ? half : 0)];
        const float2 nux0 = f2neg(f2lo(u0)), nuy0 = f2neg(f2hi(u0));
        const float2 nux1 = f2neg(f2lo(u1)), nuy1 = f2neg(f2hi(u1));
        uint32_t nx[4] = {0u, 0u, 0u, 0u};
        if (!all && w0 < w1) word(w0, nx);
        for (int w = w0; w < w1;) {
            const uint32_t c0 = nx[0], c1 = nx[1], c2 = nx[2], c3 = nx[3];
            const int we = all ? w1 : w + 1;
            if (we < w1) word(we, nx);
            if (all || __all_sync(0xffffffffu, (c0 & c1 & c2 & c3) == full_word(w)))
                np_row_bonds<false, LINEAR>(tab, g.m, 32 * w, min(S, 32 * we), P4, half, q0.bi, nux0, nuy0, nux1, nuy1,
                                            0u, 0u, 0u, 0u, Fx0, Fy0, Fx1, Fy1);
            else
                np_row_bonds<true, LINEAR>(tab, g.m, 32 * w, min(S, 32 * we), P4, half, q0.bi, nux0, nuy0, nux1, nuy1,
                                           c0, c1, c2, c3, Fx0, Fy0, Fx1, Fy1);
            w = we;
        }
    }
    // The ranges' sums in order, and the update, over all of the threads: with 4 ranges a
    // point each. The box is done with and holds the sums.
    float4 *red = P4;                         // [range][pair] {Fx, Fy}: launch_np_fast checks that it fits
    if (a.split > 1) {
        __syncthreads();
        red[sub * npairs + 2 * t] = make_float4(Fx0.x, Fx0.y, Fy0.x, Fy0.y);
        red[sub * npairs + 2 * t + 1] = make_float4(Fx1.x, Fx1.y, Fy1.x, Fy1.y);
        __syncthreads();
    }
    for (int i = a.split > 1 ? sub & 1 : 0; i < 2; i += a.split > 1 ? 2 : 1) {
        PairPts q = pair_points(g, pb, org, tile, 2 * t + i);
        if (a.split == 4) q.act[1 - sub / 2] = false;
        float2 Fx = i ? Fx1 : Fx0, Fy = i ? Fy1 : Fy0;
        if (a.split > 1) {
            float4 r = red[2 * t + i];
            Fx = f2lo(r), Fy = f2hi(r);
            for (int j = 1; j < a.split; ++j) {
                r = red[j * npairs + 2 * t + i];
                Fx = f2add(Fx, f2lo(r));
                Fy = f2add(Fy, f2hi(r));
            }
        }
        const float FA[3] = {Fx.x, Fy.x, 0.f}, FB[3] = {Fx.y, Fy.y, 0.f};
        pair_epilogue2(a, q, FA, FB, 2);
    }
}

// ---------------------------------------------------------------- dispatch

// Shared memory of pmb_fast / np_fast (base) with the stencil split over
// `split` threads per pair: the split-sum buffer (3 float2 per pair and extra part).
static size_t split_smem(const Geom &g, size_t base, int split)
{
    return base + (size_t)(split - 1) * (g.T / 2) * 3 * sizeof(float2);
}

size_t pmb_fast_smem_split(const Geom &g, int split) { return split_smem(g, pmb_fast_smem(g), split); }

// Threads per point pair: of 1, 2, 4 (at most the number of stencil words), the
// smallest that reaches the most resident threads per SM, counting the
// 1024-thread limit of 64 registers per thread and 228 KB of shared memory per
// SM (1 KB of it reserved per CTA).
static int choose_split(const Geom &g, size_t base, int pairs_per_thread = 1)
{
    const int nthr = g.T / 2 / pairs_per_thread;
    int best = 1, best_threads = 0;
    for (int split = 1; split <= 4 && split <= g.W; split *= 2) {
        const size_t smem = split_smem(g, base, split);
        if (smem > 227 * 1024) break;
        const int by_smem = (int)((228 * 1024) / (smem + 1024));
        const int ctas = std::min(by_smem, 1024 / (nthr * split));
        if (nthr * split * ctas > best_threads) {
            best = split;
            best_threads = nthr * split * ctas;
        }
    }
    return best;
}

// Ranges of stencil words in which a point pair's bonds are summed (the partial sums
// added in order), whichever kernel runs: the threads per pair of pmb_fast.
int pmb_split(const Geom &g, int pair_threads)
{
    return pair_threads ? pair_threads : choose_split(g, pmb_fast_smem(g));
}

// The stencil table as a kernel parameter when it fits one (PTAB_N float4) and
// the grid runs several waves of tiles: there the bond loops are bound by the
// shared-memory pipe that the table's reads would share (256^3 PMB step 2.43 ->
// 2.33 ms), while a grid of about one wave, bound by latency, measured slower
// with it (64^3: 0.064 -> 0.069 ms).
static bool param_table(const float4 *host, int n, int ntiles, ParamTab &tp)
{
    if (!host || n <= 0 || n > PTAB_N || ntiles < PTAB_MIN_TILES) return false;
    memcpy(tp.e, host, sizeof(float4) * (size_t)n);
    return true;
}

// Staging by columns (us a step, by pairs and by columns). With breaking, grids of two tiles
// per SM and more at m = 2 to 4 (64^3, m = 3: 57.5 and 55.0; 72 x 80 x 90 with m = 1 26.6 and 27.5,
// with m = 5 384 and 392). Below, ragged grids at m = 3 (37 x 29 x 41: 23.3 and 22.1, with breaking
// 27.1 and 24.3) and, with breaking, at m = 2 (13.4 and 12.4; without 12.5 and 12.8): m = 1 has
// few columns for the threads (9.3 and 10.6), and from m = 4 on half of the threads of a pair's
// two would wait (m = 5: 45.6 and 46.6).
static bool pmb_cols(const TileArgs &a, bool brk)
{
    const int m = a.g.m;
    if (!cols_staging(a)) return false;
    if (a.g.ntiles >= ROWS_MIN_TILES) return brk && m >= 2 && m <= 4;
    return ragged(a) && (m == 3 || (m == 2 && brk));
}

template <int DIM, bool BRK, bool SPLIT, bool COLS>
static int launch_fast_cols(const TileArgs &a, size_t smem, cudaStream_t st)
{
    PD_CUDA(smem_limit(pmb_fast<DIM, BRK, SPLIT, COLS>, smem));
    pmb_fast<DIM, BRK, SPLIT, COLS><<<a.g.ntiles, a.g.T / 2 * a.split, smem, st>>>(a);
    PD_CUDA(cudaGetLastError());
    return PD_OK;
}

template <int DIM, bool BRK, bool SPLIT>
static int launch_fast_split(const TileArgs &a, cudaStream_t st)
{
    const size_t smem = split_smem(a.g, pmb_fast_smem(a.g), a.split);
    static thread_local ParamTab tp;
    if (param_table(a.htab_a, a.ntab_a, a.g.ntiles, tp)) {
        PD_CUDA(smem_limit(pmb_fast_pt<DIM, BRK, SPLIT>, smem));
        pmb_fast_pt<DIM, BRK, SPLIT><<<a.g.ntiles, a.g.T / 2 * a.split, smem, st>>>(a, tp);
        PD_CUDA(cudaGetLastError());
        return PD_OK;
    }
    if constexpr (DIM == 3)
        if (pmb_cols(a, BRK)) return launch_fast_cols<DIM, BRK, SPLIT, true>(a, smem, st);
    return launch_fast_cols<DIM, BRK, SPLIT, false>(a, smem, st);
}

template <int DIM, bool BRK>
static int launch_fast(const TileArgs &a0, cudaStream_t st)
{
    TileArgs a = a0;
    if (a.split == 0) {
        a.split = choose_split(a.g, pmb_fast_smem(a.g));
        // with breaking a thread records its words with decisions pending in 32 bits
        while (BRK && (a.g.W + a.split - 1) / a.split > 32 && 2 * a.split <= std::min(4, a.g.W)) a.split *= 2;
    }
    if (a.split > a.g.W || split_smem(a.g, pmb_fast_smem(a.g), a.split) > 227 * 1024 || a.g.T / 2 * a.split > 1024 ||
        (BRK && (a.g.W + a.split - 1) / a.split > 32)) {
        set_error("pair_threads = %d: more than the %d stencil words, more than 32 words per thread with "
                  "breaking, or the CTA exceeds its limits", a.split, a.g.W);
        return PD_EINVAL;
    }
    if (DIM == 3 && !BRK && a.rows && rows_pmb(a.g)) return launch_rows_pmb(a, a.rows[1], st);
    return a.split > 1 ? launch_fast_split<DIM, BRK, true>(a, st) : launch_fast_split<DIM, BRK, false>(a, st);
}

size_t pmb_generic_smem(const Geom &g, int precision)
{
    const int HX = g.bx + 2 * g.m, HY = g.by + 2 * g.m, HZ = g.dim == 3 ? g.bz + 2 * g.m : 1;
    return (size_t)HX * HY * HZ * (precision == PD_FP64 ? sizeof(double4_32a) : sizeof(float4));
}

template <int DIM, bool LINEAR, bool SPLIT>
static int launch_np_split(const TileArgs &a, cudaStream_t st)
{
    const size_t smem = split_smem(a.g, np_fast_smem(a.g), a.split);
    PD_CUDA(smem_limit(np_fast<DIM, LINEAR, SPLIT>, smem));
    np_fast<DIM, LINEAR, SPLIT><<<a.g.ntiles, a.g.T / 2 * a.split, smem, st>>>(a);
    PD_CUDA(cudaGetLastError());
    return PD_OK;
}

template <bool LINEAR>
static int launch_np_rows(const TileArgs &a, cudaStream_t st)
{
    const size_t smem = np_fast_smem(a.g);
    PD_CUDA(smem_limit(np_rows<LINEAR>, smem));
    np_rows<LINEAR><<<a.g.ntiles, a.g.T / 4 * a.split, smem, st>>>(a);
    PD_CUDA(cudaGetLastError());
    return PD_OK;
}

template <int DIM, bool LINEAR>
static int launch_np_fast(const TileArgs &a0, cudaStream_t st)
{
    TileArgs a = a0;   // pair_threads applies to PMB only: the split is chosen here
    a.split = choose_split(a.g, np_fast_smem(a.g));
    // 2D wide horizons (the one-pair kernel would split): two pairs per thread by rows
    if (DIM == 2 && a.split > 1 && a.g.T >= 128) {
        const int split = choose_split(a.g, np_fast_smem(a.g), 2);
        const int2 r = tile_reach(a.g);
        const int box = (a.g.bx + 2 * a.g.m) * (a.g.by / 2 + 2 * a.g.m);
        if ((2 * r.x + 1) * (2 * r.y + 1) <= NP_LUT && split * a.g.T / 2 <= box) {
            a.split = split;
            return launch_np_rows<LINEAR>(a, st);
        }
    }
    return a.split > 1 ? launch_np_split<DIM, LINEAR, true>(a, st) : launch_np_split<DIM, LINEAR, false>(a, st);
}

// Every bond-based law: PMB, NP, LP.
int launch_pmb_args(const TileArgs &a, int precision, cudaStream_t st)
{
    const Geom &g = a.g;
    const bool brk = a.update_breaking && a.s_c > 0.0;
    if (precision == PD_FP32C && (a.model == PD_MODEL_NP || a.model == PD_MODEL_LP)) {
        const bool lin = a.model == PD_MODEL_LP;
        if (g.dim == 3) return lin ? launch_np_fast<3, true>(a, st) : launch_np_fast<3, false>(a, st);
        return lin ? launch_np_fast<2, true>(a, st) : launch_np_fast<2, false>(a, st);
    }
    if (precision == PD_FP32C) {
        if (g.dim == 3) return brk ? launch_fast<3, true>(a, st) : launch_fast<3, false>(a, st);
        return brk ? launch_fast<2, true>(a, st) : launch_fast<2, false>(a, st);
    }
    return launch_f64_bonds(a, pmb_generic_smem(g, precision), st);
}

}  // namespace pdk
