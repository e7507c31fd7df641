// pd_rows.cuh -- the FP32C passes of 3D lattices on 2^9-point (8 x 8 x 8) tiles,
// walking the stencil row by row: the PMB force + update without breaking (Eq.
// (3)) and the two LPS passes (Eq. (4), Algorithm 2), one tile per CTA of 256
// threads, one point pair (z, z + 4) per thread as in pd_pair.cuh.
//
// The stencil's rows (dz, dy fixed, dx ascending: the stencil's own order) are cut
// into segments of 5, 3 and 1 bonds with unrolled bodies, whose neighbours lie at
// consecutive box entries (immediate offsets) and share dy and dz in registers. The
// per-bond arithmetic and every point's order of summation are those of pmb_word,
// lps_dil_word and lps_force_word, so the sums are the same bits; a stencil summed
// in two ranges of words, added in order, is summed in the same two here, one after
// the other in one thread.
//
// What bounds it. Measured rates of an SM: 1.96 packed FP32 and 0.50 square root or
// reciprocal instructions a cycle. Per pair-bond of a warp (a cycle of one of the
// four SM sub-partitions) that is 40 and 32 cycles for PMB, 26 and 32 for the
// dilatation, 48 and 32 for the LPS force. The word-wise kernels take 66, 52 and 78
// in their bond loops alone (128^3): their table reads (6 to 7 constant loads a bond,
// the constant pipe 55 % busy over the whole LPS force pass) and addresses, 20 of 54
// instructions, wait beside the arithmetic. Here a bond reads 3 constant pairs, no
// offset, and no address is computed.
//
// The box holds only the planes' rows that some bond reaches: plane z' = -3 is read
// by dz = -3 alone, at dx = dy = 0, so it needs 8 rows of the 14 (m = 3: 1680 entries
// of 1960, 67 instead of 78 KB for the LPS force pass, which lets three CTAs share an
// SM instead of two), and of a column only the points within the horizon of the tile
// are loaded (2104 instead of 2 x 1960 at m = 3). Where these passes run: rows_pmb,
// rows_dil and rows_frc in pd_tile.cuh.
#pragma once

#include <string.h>

#include "pd_pair.cuh"

namespace pdk {

enum RowLaw { ROW_PMB = 0, ROW_DIL = 1, ROW_FRC = 2 };

struct RowTab {
    float4 e[ROWS_PTAB];
};

// Sums of one point pair: force, or (x alone) the dilatation's.
struct RowAcc {
    float2 x, y, z;
};

// The thread's own pair: negated displacements, and LPS's a, b.
struct RowOwn {
    float2 nux, nuy, nuz, a, b;
};

// A segment of LEN bonds from box entry `at`. te: 2 float4 an entry,
//   PMB  {|d|^2 x2, R x2} {C x2, dx x2}
//   LPS  {|d| x2, |d|^2 x2} {dx x2, V_ij, -}      (dilatation: 2 dx, and 2 dy, 2 dz)
// c0, c1: the segment's bond bits of the pair's points (MASKED).
template <int LAW, bool VOL, bool MASKED, int LEN>
__device__ __forceinline__ void row_seg(const float4 *te, float2 dyy, float2 dzz, const float4 *P4, const float2 *P2,
                                        const float4 *PT, int at, const RowOwn &o, uint32_t c0, uint32_t c1, RowAcc &F)
{
#pragma unroll
    for (int e = 0; e < LEN; ++e) {
        const float4 r4 = P4[at + e], t0 = te[2 * e], t1 = te[2 * e + 1];
        const float2 ex = f2add(f2lo(r4), o.nux), ey = f2add(f2hi(r4), o.nuy), ez = f2add(P2[at + e], o.nuz);
        const bool in0 = !MASKED || ((c0 >> e) & 1u), in1 = !MASKED || ((c1 >> e) & 1u);
        if constexpr (LAW == ROW_PMB) {
            const float2 dxx = f2hi(t1);
            const float2 yx = f2add(ex, dxx), yy = f2add(ey, dyy), yz = f2add(ez, dzz);
            float2 num = f2mul(ex, f2add(yx, dxx));
            num = f2fma(ey, f2add(yy, dyy), num);
            num = f2fma(ez, f2add(yz, dzz), num);
            const float2 qq = f2add(num, f2lo(t0));
            const float2 rr = f2sqrt(qq);
            const float2 den = f2fma(qq, f2hi(t0), f2mul(rr, f2lo(t1)));
            float2 wgt = f2mul(num, f2rcp(den));               // s V_ij / |y|
            if (MASKED) {
                wgt.x = in0 ? wgt.x : 0.f;
                wgt.y = in1 ? wgt.y : 0.f;
            }
            F.x = f2fma(wgt, yx, F.x);
            F.y = f2fma(wgt, yy, F.y);
            F.z = f2fma(wgt, yz, F.z);
        } else if constexpr (LAW == ROW_DIL) {
            float2 num = f2mul(ex, f2add(ex, f2lo(t1)));
            num = f2fma(ey, f2add(ey, dyy), num);
            num = f2fma(ez, f2add(ez, dzz), num);
            float2 x = f2mul(num, f2rcp(f2add(f2sqrt(f2add(num, f2hi(t0))), f2lo(t0))));
            if (MASKED) {
                x.x = in0 ? x.x : 0.f;
                x.y = in1 ? x.y : 0.f;
            }
            if (VOL) x = f2mul(x, make_float2(t1.z, t1.z));
            F.x = f2fma(x, f2lo(t0), F.x);
        } else {
            const float4 t4 = PT[at + e];
            const float2 dxx = f2lo(t1);
            const float2 yx = f2add(ex, dxx), yy = f2add(ey, dyy), yz = f2add(ez, dzz);
            float2 num = f2mul(ex, f2add(yx, dxx));
            num = f2fma(ey, f2add(yy, dyy), num);
            num = f2fma(ez, f2add(yz, dzz), num);
            const float2 qq = f2add(num, f2hi(t0));
            const float2 rs = f2rsqrt(qq);
            const float2 x = f2mul(num, f2rcp(f2add(f2mul(qq, rs), f2lo(t0))));
            float2 gg = f2mul(f2lo(t0), f2add(o.a, f2lo(t4)));
            gg = f2fma(x, f2add(o.b, f2hi(t4)), gg);
            if (VOL) gg = f2mul(gg, make_float2(t1.z, t1.z));
            float2 wgt = f2mul(gg, rs);
            if (MASKED) {
                wgt.x = in0 ? wgt.x : 0.f;
                wgt.y = in1 ? wgt.y : 0.f;
            }
            F.x = f2fma(wgt, yx, F.x);
            F.y = f2fma(wgt, yy, F.y);
            F.z = f2fma(wgt, yz, F.z);
        }
    }
}

template <int LAW, bool VOL, bool MASKED>
__device__ __forceinline__ void row_seg_len(int len, const float4 *te, float2 dyy, float2 dzz, const float4 *P4,
                                            const float2 *P2, const float4 *PT, int at, const RowOwn &o, uint32_t c0,
                                            uint32_t c1, RowAcc &F)
{
    if (len == 5) row_seg<LAW, VOL, MASKED, 5>(te, dyy, dzz, P4, P2, PT, at, o, c0, c1, F);
    else if (len == 3) row_seg<LAW, VOL, MASKED, 3>(te, dyy, dzz, P4, P2, PT, at, o, c0, c1, F);
    else row_seg<LAW, VOL, MASKED, 1>(te, dyy, dzz, P4, P2, PT, at, o, c0, c1, F);
}

template <int LAW, bool VOL, int PARTS, bool PTAB>
__device__ __forceinline__ void rows_body(const TileArgs &a, const RowArgs &ra, int tile, const float4 *ptab)
{
    const Geom &g = a.g;
    extern __shared__ float4 smem4[];
    float4 *P4 = smem4;                                                     // {xA, xB, yA, yB}
    float4 *PT = P4 + (LAW == ROW_FRC ? ra.nbox : 0);                       // {aA, aB, bA, bB}
    float2 *P2 = reinterpret_cast<float2 *>(PT + ra.nbox);                  // {zA, zB}
    float4 *stab = PT + ra.nbox + (ra.nbox + 1) / 2;
    __shared__ int s_nbr[27], s_plane[ROWS_PLANES];
    if (LAW != ROW_PMB && threadIdx.x == 0) prefetch_tile_masks(a, tile);
    const int4 org = __ldg(&a.tile_org[tile]);
    if (!PTAB)
        for (int k = threadIdx.x; k < ra.ntab; k += blockDim.x) stab[k] = __ldg(&ra.tab[k]);
    load_nbr(a, tile, s_nbr);
    if (threadIdx.x < ROWS_PLANES) s_plane[threadIdx.x] = ra.plane[threadIdx.x];
    // thread (lx, y, z): y rows of a warp's 16 lanes 4 apart, so that an 8-byte shared
    // load of 16 lanes covers all banks (row pitch 8 + 2m); a warp has one z
    const int lx = threadIdx.x & 7, yr = (threadIdx.x >> 3) & 7, lz = threadIdx.x >> 6;
    const int ly = (yr & 1) * 4 + (yr >> 1);
    const int sA = tile * 512 + brick_code(3, lx, ly, lz), sB = sA + 256;    // z + 4: code bit 8
    // whether every bond of the warp's points is there; the loads overlap the staging's
    bool whole = true;
    for (int w = 0; w < g.W; ++w) {
        const size_t mo = (size_t)w * g.nslots;
        const int nb = min(32, g.S - 32 * w);
        whole = whole && (a.mask[mo + sA] & a.mask[mo + sB]) == (nb == 32 ? 0xffffffffu : (1u << nb) - 1u);
    }
    whole = __all_sync(0xffffffffu, whole);
    __syncthreads();
    // points loaded together: one where registers are short (64^3 PMB step 0.0479 ms with
    // two, 0.0467 with one; LPS force at three CTAs 0.334 and 0.320), else two
    stage_columns<LAW == ROW_FRC, LAW == ROW_PMB || (LAW == ROW_FRC && PTAB) ? 1 : 2>(a, org, tile_ref32(a, tile), s_nbr,
                                                                                    s_plane, P4, P2, PT);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (LAW == ROW_FRC) prefetch_tile_update(a, tile);
        if (LAW == ROW_DIL) l2_prefetch(a.minv32 + (size_t)tile * 512, 4 * 512);
    }

    const int HX = 8 + 2 * g.m, own = (lx + g.m) + HX * (ly + g.m);
    RowOwn o;
    {
        const int b = own + s_plane[lz + g.m];
        const float4 u4 = P4[b];
        o.nux = f2neg(f2lo(u4));
        o.nuy = f2neg(f2hi(u4));
        o.nuz = f2neg(P2[b]);
        if (LAW == ROW_FRC) {
            const float4 t4 = PT[b];
            o.a = f2lo(t4);
            o.b = f2hi(t4);
        }
    }
    const float4 *ent = PTAB ? ptab : stab, *seg = ent + 2 * g.S;
    const float2 zero = make_float2(0.f, 0.f);
    RowAcc F = {zero, zero, zero}, first = {zero, zero, zero};
    // segment {offset in a plane | (dz + m) << 16 | bonds << 24, first stencil entry, dy, dz}
    auto entry = [&](int bits) { return own + (int)(short)(bits & 0xffff) + s_plane[lz + ((bits >> 16) & 0xff)]; };
    if (whole) {
        float4 h = seg[0];
        for (int sg = 0; sg < ra.nseg; ++sg) {
            const float4 hn = seg[sg + 1];              // (a segment of zeros ends the table)
            if (PARTS == 2 && sg == ra.split) {
                first = F;
                F = {zero, zero, zero};
            }
            const int b = __float_as_int(h.x);
            row_seg_len<LAW, VOL, false>(b >> 24, ent + 2 * __float_as_int(h.y), make_float2(h.z, h.z),
                                         make_float2(h.w, h.w), P4, P2, PT, entry(b), o, 0u, 0u, F);
            h = hn;
        }
    } else {
        int wc = 0;
        auto word = [&](int w, int s) { return w < g.W ? a.mask[(size_t)w * g.nslots + s] : 0u; };
        uint32_t l0 = word(0, sA), l1 = word(0, sB), h0 = word(1, sA), h1 = word(1, sB);
        uint32_t n0 = word(2, sA), n1 = word(2, sB);
        for (int sg = 0; sg < ra.nseg; ++sg) {
            const float4 h = seg[sg];
            if (PARTS == 2 && sg == ra.split) {
                first = F;
                F = {zero, zero, zero};
            }
            const int b = __float_as_int(h.x), k = __float_as_int(h.y);
            if ((k >> 5) != wc) {           // segments follow one another: the next word
                ++wc;
                l0 = h0;
                l1 = h1;
                h0 = n0;
                h1 = n1;
                n0 = word(wc + 2, sA);
                n1 = word(wc + 2, sB);
            }
            row_seg_len<LAW, VOL, true>(b >> 24, ent + 2 * k, make_float2(h.z, h.z), make_float2(h.w, h.w), P4, P2, PT,
                                        entry(b), o, __funnelshift_r(l0, h0, k & 31), __funnelshift_r(l1, h1, k & 31),
                                        F);
        }
    }
    RowAcc tot = F;
    if (PARTS == 2) {
        tot.x = f2add(first.x, F.x);
        tot.y = f2add(first.y, F.y);
        tot.z = f2add(first.z, F.z);
    }
    PairPts q;
    q.slot[0] = sA;
    q.slot[1] = sB;
    const bool inxy = org.x + lx < g.nx && org.y + ly < g.ny;
    q.act[0] = inxy && org.z + lz < g.nz;
    q.act[1] = inxy && org.z + lz + 4 < g.nz;
    q.bi = 0;
    if constexpr (LAW == ROW_DIL) {
        if (q.act[0]) a.theta32[sA] = 3.f * __ldg(&a.minv32[sA]) * tot.x.x;
        if (q.act[1]) a.theta32[sB] = 3.f * __ldg(&a.minv32[sB]) * tot.x.y;
    } else {
        const float FA[3] = {tot.x.x, tot.y.x, tot.z.x}, FB[3] = {tot.x.y, tot.y.y, tot.z.y};
        pair_epilogue2(a, q, FA, FB, 3);
    }
}

}  // namespace pdk
