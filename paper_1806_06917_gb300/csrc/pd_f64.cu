// pd_f64.cu -- the all-FP64 passes (PD_FP64): the bond-based force + update with
// breaking (Eq. (3), Algorithm 1), the LPS dilatation and force + update (Eq. (4),
// Algorithm 2), and the tangent product of Eq. (6) and its adjoint.
//
// What bounds them. An SM issues one FP64 warp instruction every 16.6 cycles (measured:
// 0.060 a cycle), 64 times less than FP32, so the passes cost their FP64 instructions and
// everything else hides behind them. The generic templates spent about 65 a bond on PMB and
// 115 on the two LPS passes, half of them in the correctly rounded 1 / sqrt and the
// divisions (and, in 2D, on a third component of zeros). Here a bond takes, in lattice
// units (xi = d, e = eta, y = d + e, r0 = |d|, r = |y|):
//   num = 2 d.e + e.e, q = r0^2 + num                                     3 + 6 + 1
//   r   = sqrt(q): the rsqrt.approx.ftz.f64 seed (21 bits) and one third-order
//         step, z = q y0, g = 1 - z y0, r = z + z g (1/2 + 3/8 g)                   5
//   w   = num / (R q + C r), R = r0 / V_ij, C = r0^2 / V_ij: s V_ij / r in
//         one quotient, z = num y0 from rcp.approx.ftz.f64 and its residual
//         over den, z + (num - den z) y0 (2 - den y0)                          2 + 5
//   F  += w y                                                                 3 + 3
// 28 in 3D and 23 in 2D (dilatation 23, LPS force 32, tangent product 45 and 36). The
// quotient, the dilatation's root and 1 / sqrt(q) round once. 64^3 PMB step with breaking
// 3.58 -> 1.67 ms (28 instructions a bond cost 1.45), 40^3 LPS step 1.70 -> 0.88 ms, 97^2
// NP step (m = 8; its exponential by a short series near 0) 2.06 -> 0.165 ms, tangent product
// and force of the 200^2 plate through the torch bridge 0.556 -> 0.25 ms. The error against
// extended precision is that of the templates, 1.3 to 5e-16 for m = 1 to 5 (relative L2), also
// for compressed bonds (f64_len2).
#include <algorithm>
#include <type_traits>

#include "pd_tile.cuh"

namespace pdk {

// num = |y|^2 - |d|^2 = 2 d.e + e.e (dx..: 2 d): the small squares first, so that they round
// below the other terms, whose products are exact where d has the sides 1 and 2.
__device__ __forceinline__ double f64_num2(const F64Ent &e, double ex, double ey)
{
    return fma(e.dy, ey, fma(e.dx, ex, fma(ey, ey, ex * ex)));
}
__device__ __forceinline__ double f64_num3(const F64Ent &e, double ex, double ey, double ez)
{
    return fma(e.dz, ez, fma(e.dy, ey, fma(e.dx, ex, fma(ez, ez, fma(ey, ey, ex * ex)))));
}

// Box geometry and the thread's point.
struct F64Pt {
    int slot, bi, x, y, z;
    bool act;
};

template <int DIM>
__device__ __forceinline__ F64Pt f64_point(const Geom &g, const int4 &org, int tile, int t, int HX, int HY)
{
    const int lx = t & (g.bx - 1), ly = (t >> g.lbx) & (g.by - 1), lz = DIM == 3 ? t >> (g.lbx + g.lby) : 0;
    F64Pt p;
    p.slot = tile * g.T + brick_code(DIM, lx, ly, lz);
    p.x = org.x + lx;
    p.y = org.y + ly;
    p.z = org.z + lz;
    p.act = p.x < g.nx && p.y < g.ny && p.z < g.nz;
    p.bi = (lx + g.m) + HX * ((ly + g.m) + HY * (DIM == 3 ? lz + g.m : 0));
    return p;
}

// exp(x) for x <= 0 (the NP law's exponent): near 0, where small strains keep it, by
// the series to x^7 / 7!, whose remainder is below 2^-53 for |x| < 2^-6.
__device__ __forceinline__ double f64_exp_neg(double x)
{
    if (!(x > -0x1p-6)) return exp(x);
    double p = 1.0 / 5040.0;
    p = fma(p, x, 1.0 / 720.0);
    p = fma(p, x, 1.0 / 120.0);
    p = fma(p, x, 1.0 / 24.0);
    p = fma(p, x, 1.0 / 6.0);
    p = fma(p, x, 0.5);
    p = fma(p, x, 1.0);
    return fma(p, x, 1.0);
}

// |y|^2 of a bond with lattice vector d, |d|^2 = d2: num + d2, and y.y where a bond has
// lost half of that and more. There the sum cancels (relative error 2^-53 d2 / |y|^2: 1e-12
// at a hundredth of the length, and down to 0 or below for a collapsed bond); above, both
// agree to the last bit or two. High words are compared as integers, so that only the
// bonds concerned pay FP64 instructions (y.y in line was predicated, and every bond paid:
// 64^3 PMB step 1.64 -> 1.81 ms): in the PMB pass y.y stands out of line; the LPS passes and
// the tangent product sum a mask word's bonds with num + d2, note whether one is so short,
// and then sum the word once more with EXACT, which leaves the loop without a branch (40^3
// LPS step 0.928 -> 0.880 ms against the call; PMB, whose breaking test is a call as it is, 64^3
// with m = 4 3.48 -> 3.60).
__device__ __forceinline__ bool f64_short(double q, double d2) { return __double2hiint(q) < __double2hiint(d2) - 0x100000; }
__device__ __noinline__ double f64_dot(double x, double y, double z) { return fma(z, z, fma(y, y, x * x)); }
__device__ __forceinline__ double f64_len2(double num, double d2, double yx, double yy, double yz)
{
    const double q = num + d2;
    return f64_short(q, d2) ? f64_dot(yx, yy, yz) : q;
}
template <bool EXACT>
__device__ __forceinline__ double f64_len2(double num, double d2, double yx, double yy, double yz, bool &low)
{
    double q = num + d2;
    if (!EXACT) low = low || f64_short(q, d2);
    else if (f64_short(q, d2)) q = fma(yz, yz, fma(yy, yy, yx * yx));
    return q;
}

// ------------------------------------------------------------- bond-based

// The FP64 stretch of bond (si, sj) with lattice offset d from the global FP64
// staging (the FP64 path's u), bitwise the same from both ends of the bond.
__device__ __forceinline__ double canon_stretch64(const TileArgs &a, int si, int sj, double dx, double dy, double dz,
                                                  double d2)
{
    const double4_32a ui = a.src_d4[si], uj = a.src_d4[sj];
    const double ex = __dmul_rn(__dsub_rn(uj.x, ui.x), a.inv_h);
    const double ey = __dmul_rn(__dsub_rn(uj.y, ui.y), a.inv_h);
    const double ez = __dmul_rn(__dsub_rn(uj.z, ui.z), a.inv_h);
    double num = __dmul_rn(ex, __dadd_rn(__dadd_rn(ex, dx), dx));
    num = __fma_rn(ey, __dadd_rn(__dadd_rn(ey, dy), dy), num);
    num = __fma_rn(ez, __dadd_rn(__dadd_rn(ez, dz), dz), num);
    const double r0 = __dsqrt_rn(d2), r = __dsqrt_rn(__dadd_rn(num, d2));
    return __ddiv_rn(num, __dmul_rn(r0, __dadd_rn(r, r0)));
}

// Whether a bond breaks (s > s_c): decided from s = num / (r0 (r + r0)), and within
// 2^-30 of s_c from both points' global state (canon_stretch64). Out of line: reached
// only by bonds whose num lies above F64Ent::near (s > s_c exactly when num > r0^2
// ((1 + s_c)^2 - 1); the loop compares high words, as integers).
__device__ __noinline__ bool f64_breaks(const TileArgs *ap, int slot, int x, int y, int z, const F64Ent *e, double num)
{
    const TileArgs &a = *ap;
    const double r0 = sqrt(e->d2), r = sqrt(e->d2 + num);
    const double s = num / (r0 * (r + r0));
    if (fabs(s - a.s_c) <= 0x1p-30 * a.s_c) {
        const double dx = 0.5 * e->dx, dy = 0.5 * e->dy, dz = 0.5 * e->dz;
        const int sj = slot_at(a.g, a.tile_lut, x + (int)dx, y + (int)dy, z + (int)dz);
        return sj >= 0 && canon_stretch64(a, slot, sj, dx, dy, dz, e->d2) > a.s_c;
    }
    return s > a.s_c;
}

template <int DIM, bool BRK>
__global__ void __launch_bounds__(256) f64_pmb(const __grid_constant__ TileArgs a)
{
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const Geom &g = a.g;
    const int m = g.m, HX = g.bx + 2 * m, HY = g.by + 2 * m, HZ = DIM == 3 ? g.bz + 2 * m : 1;
    const F64Ent *tab = a.tab64;
    double4_32a *box = reinterpret_cast<double4_32a *>(smem_raw);
    const int tile = blockIdx.x;
    const int4 org = __ldg(&a.tile_org[tile]);
    stage_box64(box, HX, HY, HX * HY * HZ, m, a, org, tile_ref64(a, tile), a.inv_h);
    __syncthreads();
    for (int t = threadIdx.x; t < g.T; t += blockDim.x) {
        const F64Pt p = f64_point<DIM>(g, org, tile, t, HX, HY);
        if (!p.act) continue;
        const double4_32a ui = box[p.bi];
        double Fx = 0.0, Fy = 0.0, Fz = 0.0;
        for (int w = 0; w < g.W; ++w) {
            const uint32_t word = a.mask[(size_t)w * g.nslots + p.slot];
            uint32_t nword = word;
            const int nb = min(32, g.S - 32 * w);
#pragma unroll 4
            for (int b = 0; b < nb; ++b) {
                if (!((word >> b) & 1u)) continue;
                const F64Ent &e = tab[32 * w + b];
                const double4_32a rj = box[p.bi + e.off];
                const double ex = rj.x - ui.x, ey = rj.y - ui.y;
                const double yx = fma(0.5, e.dx, ex), yy = fma(0.5, e.dy, ey);
                double num, yz = 0.0;
                if (DIM == 3) {
                    const double ez = rj.z - ui.z;
                    yz = fma(0.5, e.dz, ez);
                    num = f64_num3(e, ex, ey, ez);
                } else {
                    num = f64_num2(e, ex, ey);
                }
                if (BRK && __double2hiint(num) >= e.near &&
                    f64_breaks(&a, p.slot, p.x, p.y, p.z, &e, num)) {
                    nword &= ~(1u << b);
                    continue;
                }
                const double q = f64_len2(num, e.d2, yx, yy, yz);
                const double wgt = f64_div(num, fma(e.C, f64_sqrt(q), e.R * q));
                Fx = fma(wgt, yx, Fx);
                Fy = fma(wgt, yy, Fy);
                if (DIM == 3) Fz = fma(wgt, yz, Fz);
            }
            if (BRK && nword != word) a.mask[(size_t)w * g.nslots + p.slot] = nword;
        }
        const double f[3] = {a.cV * Fx, a.cV * Fy, a.cV * Fz};
        point_epilogue(a, p.slot, f, DIM, true);
    }
}

// NP / LP (Algorithm 1): with p = d.e the bond term is k p [exp(a' p^2) for NP] d.
template <int DIM, bool LINEAR>
__global__ void __launch_bounds__(256) f64_np(const __grid_constant__ TileArgs a)
{
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const Geom &g = a.g;
    const int m = g.m, HX = g.bx + 2 * m, HY = g.by + 2 * m, HZ = DIM == 3 ? g.bz + 2 * m : 1;
    const F64Ent *tab = a.tab64;
    double4_32a *box = reinterpret_cast<double4_32a *>(smem_raw);
    const int tile = blockIdx.x;
    const int4 org = __ldg(&a.tile_org[tile]);
    stage_box64(box, HX, HY, HX * HY * HZ, m, a, org, tile_ref64(a, tile), a.inv_h);
    __syncthreads();
    for (int t = threadIdx.x; t < g.T; t += blockDim.x) {
        const F64Pt p = f64_point<DIM>(g, org, tile, t, HX, HY);
        if (!p.act) continue;
        const double4_32a ui = box[p.bi];
        double Fx = 0.0, Fy = 0.0, Fz = 0.0;
        for (int w = 0; w < g.W; ++w) {
            const uint32_t word = a.mask[(size_t)w * g.nslots + p.slot];
            const int nb = min(32, g.S - 32 * w);
#pragma unroll 4
            for (int b = 0; b < nb; ++b) {
                if (!((word >> b) & 1u)) continue;
                const F64Ent &e = tab[32 * w + b];
                const double4_32a rj = box[p.bi + e.off];
                double dot = (rj.x - ui.x) * e.dx;
                dot = fma(rj.y - ui.y, e.dy, dot);
                if (DIM == 3) dot = fma(rj.z - ui.z, e.dz, dot);
                double wgt = e.R * dot;
                if (!LINEAR) wgt *= f64_exp_neg(e.C * (dot * dot));
                Fx = fma(wgt, e.dx, Fx);
                Fy = fma(wgt, e.dy, Fy);
                if (DIM == 3) Fz = fma(wgt, e.dz, Fz);
            }
        }
        const double f[3] = {a.cV * Fx, a.cV * Fy, a.cV * Fz};
        point_epilogue(a, p.slot, f, DIM, true);
    }
}

// ------------------------------------------------------------------- LPS

template <bool VOL>
__global__ void __launch_bounds__(256) f64_lps_dil(const __grid_constant__ TileArgs a)
{
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const Geom &g = a.g;
    const int m = g.m, HX = g.bx + 2 * m, HY = g.by + 2 * m, HZ = g.bz + 2 * m;
    const F64Ent *tab = a.tab64;
    double4_32a *box = reinterpret_cast<double4_32a *>(smem_raw);
    const int tile = blockIdx.x;
    const int4 org = __ldg(&a.tile_org[tile]);
    stage_box64(box, HX, HY, HX * HY * HZ, m, a, org, tile_ref64(a, tile), a.inv_h);
    __syncthreads();
    for (int t = threadIdx.x; t < g.T; t += blockDim.x) {
        const F64Pt p = f64_point<3>(g, org, tile, t, HX, HY);
        if (!p.act) continue;
        const double4_32a ui = box[p.bi];
        double acc = 0.0;
        for (int w = 0; w < g.W; ++w) {
            const uint32_t word = a.mask[(size_t)w * g.nslots + p.slot];
            const int nb = min(32, g.S - 32 * w);
            const double acc0 = acc;
            bool low = false;
            auto bond = [&](int b, auto exact) {
                const F64Ent &e = tab[32 * w + b];
                const double4_32a rj = box[p.bi + e.off];
                const double ex = rj.x - ui.x, ey = rj.y - ui.y, ez = rj.z - ui.z;
                const double num = f64_num3(e, ex, ey, ez);
                const double q = f64_len2<exact.value>(num, e.d2, fma(0.5, e.dx, ex), fma(0.5, e.dy, ey),
                                                       fma(0.5, e.dz, ez), low);
                double x = f64_div(num, f64_sqrt_rn(q) + e.R);
                if (VOL) x *= e.C;
                acc = fma(e.R, x, acc);
            };
#pragma unroll 4
            for (int b = 0; b < nb; ++b) {
                if (!((word >> b) & 1u)) continue;
                bond(b, std::false_type());
            }
            if (low) {
                acc = acc0;
#pragma unroll 1
                for (int b = 0; b < nb; ++b)
                    if ((word >> b) & 1u) bond(b, std::true_type());
            }
        }
        a.theta64[p.slot] = 3.0 * acc / a.mtil[p.slot];
    }
}

template <bool VOL>
__global__ void __launch_bounds__(256) f64_lps_force(const __grid_constant__ TileArgs a)
{
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const Geom &g = a.g;
    const int m = g.m, HX = g.bx + 2 * m, HY = g.by + 2 * m, HZ = g.bz + 2 * m, nbox = HX * HY * HZ;
    const F64Ent *tab = a.tab64;
    double4_32a *box = reinterpret_cast<double4_32a *>(smem_raw);    // u, (3K - 5mu) theta / m~
    double *boxb = reinterpret_cast<double *>(box + nbox);                              // 15mu / m~
    const int tile = blockIdx.x;
    const int4 org = __ldg(&a.tile_org[tile]);
    const double3 ref = tile_ref64(a, tile);
    for (int b = threadIdx.x; b < nbox; b += blockDim.x) {
        int x, y, z;
        box_coord(b, HX, HY, m, 3, org, x, y, z);
        const int s = slot_at(g, a.tile_lut, x, y, z);
        double4_32a r = make_double4_32a(0.0, 0.0, 0.0, 0.0);
        double rb = 0.0;
        if (s >= 0) {
            const double4_32a d = a.src_d4[s];
            r.x = (d.x - ref.x) * a.inv_h;
            r.y = (d.y - ref.y) * a.inv_h;
            r.z = (d.z - ref.z) * a.inv_h;
            const double mi = f64_div(1.0, a.mtil[s]);
            r.w = a.A * (a.theta64[s] * mi);
            rb = a.B * mi;
        }
        box[b] = r;
        boxb[b] = rb;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < g.T; t += blockDim.x) {
        const F64Pt p = f64_point<3>(g, org, tile, t, HX, HY);
        if (!p.act) continue;
        const double4_32a ui = box[p.bi];
        const double bi = boxb[p.bi];
        double Fx = 0.0, Fy = 0.0, Fz = 0.0;
        for (int w = 0; w < g.W; ++w) {
            const uint32_t word = a.mask[(size_t)w * g.nslots + p.slot];
            const int nb = min(32, g.S - 32 * w);
            const double X0 = Fx, Y0 = Fy, Z0 = Fz;
            bool low = false;
            auto bond = [&](int b, auto exact) {
                const F64Ent &e = tab[32 * w + b];
                const int bj = p.bi + e.off;
                const double4_32a rj = box[bj];
                const double ex = rj.x - ui.x, ey = rj.y - ui.y, ez = rj.z - ui.z;
                const double yx = fma(0.5, e.dx, ex), yy = fma(0.5, e.dy, ey), yz = fma(0.5, e.dz, ez);
                const double num = f64_num3(e, ex, ey, ez);
                const double q = f64_len2<exact.value>(num, e.d2, yx, yy, yz, low), rs = f64_rsqrt(q);
                const double x = f64_div(num, fma(q, rs, e.R));
                double gg = e.R * (ui.w + rj.w);
                gg = fma(x, bi + boxb[bj], gg);
                double wgt = gg * rs;
                if (VOL) wgt *= e.C;
                Fx = fma(wgt, yx, Fx);
                Fy = fma(wgt, yy, Fy);
                Fz = fma(wgt, yz, Fz);
            };
#pragma unroll 4
            for (int b = 0; b < nb; ++b) {
                if (!((word >> b) & 1u)) continue;
                bond(b, std::false_type());
            }
            if (low) {
                Fx = X0, Fy = Y0, Fz = Z0;
#pragma unroll 1
                for (int b = 0; b < nb; ++b)
                    if ((word >> b) & 1u) bond(b, std::true_type());
            }
        }
        const double f[3] = {a.inv_h * Fx, a.inv_h * Fy, a.inv_h * Fz};
        point_epilogue(a, p.slot, f, 3, true);
    }
}

// --------------------------------------------------------------- tangent

// (K w)_i = (c V / h) sum_j V_ij [ (n.dw) (1 / |d| - s / r) n + (s / r) dw ], n = y / r. The
// coefficient of n n^T is 1 / r as well, but rs^3 y.dw y carries the root's rounding three
// times (2D, m = 2: 1.74e-16 against 1.60e-16). D_ij is symmetric and the volumes are
// uniform, so the adjoint's transposed gather evaluates the same terms.
template <int DIM>
__global__ void __launch_bounds__(256) f64_jvp(const __grid_constant__ TileArgs a)
{
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const Geom &g = a.g;
    const int m = g.m, HX = g.bx + 2 * m, HY = g.by + 2 * m, HZ = DIM == 3 ? g.bz + 2 * m : 1, nbox = HX * HY * HZ;
    const F64Ent *tab = a.tab64;
    double4_32a *box = reinterpret_cast<double4_32a *>(smem_raw);
    double4_32a *wbox = box + nbox;
    const int tile = blockIdx.x;
    const int4 org = __ldg(&a.tile_org[tile]);
    stage_box64(box, HX, HY, nbox, m, a, org, tile_ref64(a, tile), a.inv_h);
    const int rs_slot = __ldg(&a.tile_ref[tile]);
    const double wr[3] = {a.w[0][rs_slot], a.w[1][rs_slot], DIM == 3 ? a.w[2][rs_slot] : 0.0};
    for (int b = threadIdx.x; b < nbox; b += blockDim.x) {
        int x, y, z;
        box_coord(b, HX, HY, m, DIM, org, x, y, z);
        const int s = slot_at(g, a.tile_lut, x, y, z);
        double4_32a r = make_double4_32a(0.0, 0.0, 0.0, 0.0);
        if (s >= 0) {
            r.x = a.w[0][s] - wr[0];
            r.y = a.w[1][s] - wr[1];
            if (DIM == 3) r.z = a.w[2][s] - wr[2];
        }
        wbox[b] = r;
    }
    __syncthreads();
    const double sc = a.cV * a.inv_h;
    for (int t = threadIdx.x; t < g.T; t += blockDim.x) {
        const F64Pt p = f64_point<DIM>(g, org, tile, t, HX, HY);
        if (!p.act) continue;
        const double4_32a ui = box[p.bi], wi = wbox[p.bi];
        double ox = 0.0, oy = 0.0, oz = 0.0;
        for (int w = 0; w < g.W; ++w) {
            const uint32_t word = a.mask[(size_t)w * g.nslots + p.slot];
            const int nb = min(32, g.S - 32 * w);
            const double X0 = ox, Y0 = oy, Z0 = oz;
            bool low = false;
            auto bond = [&](int b, auto exact) {
                const F64Ent &e = tab[32 * w + b];
                const double4_32a uj = box[p.bi + e.off], wj = wbox[p.bi + e.off];
                const double ex = uj.x - ui.x, ey = uj.y - ui.y;
                const double yx = fma(0.5, e.dx, ex), yy = fma(0.5, e.dy, ey);
                const double dwx = wj.x - wi.x, dwy = wj.y - wi.y;
                double ndw = yx * dwx;
                ndw = fma(yy, dwy, ndw);
                double num, yz = 0.0, dwz = 0.0;
                if (DIM == 3) {
                    const double ez = uj.z - ui.z;
                    yz = fma(0.5, e.dz, ez);
                    num = f64_num3(e, ex, ey, ez);
                    dwz = wj.z - wi.z;
                    ndw = fma(yz, dwz, ndw);
                } else {
                    num = f64_num2(e, ex, ey);
                }
                const double q = f64_len2<exact.value>(num, e.d2, yx, yy, yz, low), rs = f64_rsqrt(q);
                const double cs = f64_div(num, fma(e.C, q * rs, e.R * q));         // V_ij s / r
                const double cn = ndw * rs * (e.I - cs) * rs;                      // times y
                // a bond's two terms first: added to the sum one by one they round it twice (an
                // error of 3.7e-16 against 2.7e-16, m = 5 in 2D)
                ox += fma(cn, yx, cs * dwx);
                oy += fma(cn, yy, cs * dwy);
                if (DIM == 3) oz += fma(cn, yz, cs * dwz);
            };
#pragma unroll 2
            for (int b = 0; b < nb; ++b) {
                if (!((word >> b) & 1u)) continue;
                bond(b, std::false_type());
            }
            if (low) {
                ox = X0, oy = Y0, oz = Z0;
#pragma unroll 1
                for (int b = 0; b < nb; ++b)
                    if ((word >> b) & 1u) bond(b, std::true_type());
            }
        }
        a.jv[0][p.slot] = sc * ox;
        a.jv[1][p.slot] = sc * oy;
        if (DIM == 3) a.jv[2][p.slot] = sc * oz;
    }
}

// ---------------------------------------------------------------- launches

template <class K>
static int go(K *k, const TileArgs &a, size_t smem, cudaStream_t st)
{
    PD_CUDA(smem_limit(k, smem));
    k<<<a.g.ntiles, std::min(256, a.g.T), smem, st>>>(a);
    PD_CUDA(cudaGetLastError());
    return PD_OK;
}

int launch_f64_bonds(const TileArgs &a, size_t smem, cudaStream_t st)
{
    const bool d3 = a.g.dim == 3;
    if (a.model == PD_MODEL_NP) return d3 ? go(f64_np<3, false>, a, smem, st) : go(f64_np<2, false>, a, smem, st);
    if (a.model == PD_MODEL_LP) return d3 ? go(f64_np<3, true>, a, smem, st) : go(f64_np<2, true>, a, smem, st);
    if (a.update_breaking && a.s_c > 0.0)
        return d3 ? go(f64_pmb<3, true>, a, smem, st) : go(f64_pmb<2, true>, a, smem, st);
    return d3 ? go(f64_pmb<3, false>, a, smem, st) : go(f64_pmb<2, false>, a, smem, st);
}

int launch_f64_lps(const TileArgs &a, int dil, size_t smem, cudaStream_t st)
{
    if (dil) return a.vol_corr ? go(f64_lps_dil<true>, a, smem, st) : go(f64_lps_dil<false>, a, smem, st);
    return a.vol_corr ? go(f64_lps_force<true>, a, smem, st) : go(f64_lps_force<false>, a, smem, st);
}

int launch_f64_jvp(const TileArgs &a, size_t smem, cudaStream_t st)
{
    return a.g.dim == 3 ? go(f64_jvp<3>, a, smem, st) : go(f64_jvp<2>, a, smem, st);
}

}  // namespace pdk
