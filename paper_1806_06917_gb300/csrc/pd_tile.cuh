// pd_tile.cuh -- machinery shared by the tile kernels (force, step, tangent,
// energy): FP64 roots and quotients, shared-memory staging of a tile's halo box,
// the rules of the dispatch and the kernels' arguments.
//
// A CTA owns one tile (a Morton brick of T = 2^L lattice points). It stages the
// displacements of the brick plus an m-wide halo into shared memory as a dense
// box in lattice coordinates, so the neighbour at stencil offset d of the point
// at box index b sits at box index b + d.x + HX (d.y + HY d.z): one
// conflict-free vector load per bond. Displacements are staged in lattice units
// relative to a per-tile reference displacement,
//     u~_j = (u_j - u_ref) / h,
// formed from FP32 hi/lo pairs (FP32C) or FP64 (FP64 path). Bond vectors are
// then eta = u~_j - u~_i and xi = d (integers), so the cancellation that a
// rigid translation or a large displacement would cause in FP32 never occurs:
// the error of eta is relative to the variation of u across one halo box.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"

// float4 words per stencil entry of the FP32C NP / LP table (np_word in
// pd_force_pmb.cu; built in pd_api.cu)
#define NP_TAB_WORDS(dim) ((dim) == 3 ? 3 : 2)

namespace pdk {

// ------------------------------------------------------------ FP64 helpers

__device__ __forceinline__ double seed_rsqrt(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
__device__ __forceinline__ double seed_rcp(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}

// The seeds carry 21 significant bits (their low words are zero), so the products marked
// exact are. sqrt(q) for q > 0: one third-order (Halley-type) step from the seed; the
// rounding of z is left in the result (below 0.8 ulp).
__device__ __forceinline__ double f64_sqrt(double q)
{
    const double y = seed_rsqrt(q), z = q * y;
    const double g = fma(-z, y, 1.0);
    return fma(z * g, fma(0.375, g, 0.5), z);
}

// The same with the residual of z: nothing is left but the last rounding.
__device__ __forceinline__ double f64_sqrt_rn(double q)
{
    const double y = seed_rsqrt(q), z = q * y;
    const double p = fma(-z, z, q) * y, g = p * y;
    return fma(p, fma(0.375, g, 0.5), z);
}

// 1 / sqrt(q) the same way (y y is exact).
__device__ __forceinline__ double f64_rsqrt(double q)
{
    const double y = seed_rsqrt(q);
    const double g = fma(-q, y * y, 1.0);
    return fma(y * g, fma(0.375, g, 0.5), y);
}

// a / b for b in the normal range: the quotient a y and its residual, divided by the seed
// corrected once. The last rounding alone is left (without the residual, the rounding of
// a y is too: 1 ulp).
__device__ __forceinline__ double f64_div(double a, double b)
{
    const double y = seed_rcp(b), z = a * y;
    return fma(fma(-b, z, a), fma(y, fma(-b, y, 1.0), y), z);
}

// 1/sqrt(q) and a/b of the templates: hardware approximations in FP32 (a few ulp), in FP64
// the steps above, which round once each (1.0 / sqrt(q) twice) at a third of the
// instructions (energies of the 200^2 plate 292 -> 185 us, 400^2 solve of 60 steps with m = 8
// 738 -> 706 us a step).
__device__ __forceinline__ float prsqrt1(float q) { return rsqrtf(q); }
__device__ __forceinline__ double prsqrt1(double q) { return f64_rsqrt(q); }
__device__ __forceinline__ float pdiv1(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double pdiv1(double a, double b) { return f64_div(a, b); }

// ------------------------------------------------------------------ stencil

// Offsets of the horizon stencil {d : 0 < |d|^2 <= m^2}, which is ordered by (dz, dy, dx)
// ascending.
__host__ __device__ constexpr int stencil_size(int dim, int m)
{
    int idx = 0;
    for (int dz = (dim == 3 ? -m : 0); dz <= (dim == 3 ? m : 0); ++dz)
        for (int dy = -m; dy <= m; ++dy)
            for (int dx = -m; dx <= m; ++dx) {
                int d2 = dx * dx + dy * dy + dz * dz;
                if (d2 != 0 && d2 <= m * m) ++idx;
            }
    return idx;
}

// Partial-volume factor in lattice units: (m + 1/2 - |d|) for |d| > m - 1/2.
__host__ __device__ constexpr double vol_factor_lattice(int m, double r0)
{
    return r0 > m - 0.5 ? (m + 0.5 - r0) : 1.0;
}

// --------------------------------------------------------------- staging

// Global coordinates of box index b for a tile with origin org (runtime box dims).
__device__ __forceinline__ void box_coord(int b, int HX, int HY, int m, int dim, const int4 &org,
                                          int &x, int &y, int &z)
{
    int bxl = b % HX;
    int rest = b / HX;
    int byl = rest % HY;
    int bzl = rest / HY;
    x = org.x + bxl - m;
    y = org.y + byl - m;
    z = dim == 3 ? org.z + bzl - m : 0;
}

// --------------------------------------------------------- slot lookup

// Spread the bits of x so that bit b moves to bit 3b (x < 1024) or 2b (x < 65536).
__device__ __forceinline__ uint32_t spread3(uint32_t x)
{
    x = (x | (x << 16)) & 0x030000FFu;
    x = (x | (x << 8)) & 0x0300F00Fu;
    x = (x | (x << 4)) & 0x030C30C3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}
__device__ __forceinline__ uint32_t spread2(uint32_t x)
{
    x = (x | (x << 8)) & 0x00FF00FFu;
    x = (x | (x << 4)) & 0x0F0F0F0Fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
    return x;
}

// Local Morton code of brick-local coordinates.
__device__ __forceinline__ int brick_code(int dim, int x, int y, int z)
{
    return dim == 3 ? (int)(spread3(x) | (spread3(y) << 1) | (spread3(z) << 2))
                    : (int)(spread2(x) | (spread2(y) << 1));
}

// Slot of lattice point (x, y, z), or -1 outside the grid.
__device__ __forceinline__ int slot_at(const Geom &g, const int *tile_lut, int x, int y, int z)
{
    if ((unsigned)x >= (unsigned)g.nx || (unsigned)y >= (unsigned)g.ny || (unsigned)z >= (unsigned)g.nz)
        return -1;
    int tx = x >> g.lbx, ty = y >> g.lby, tz = z >> g.lbz;
    int t = __ldg(&tile_lut[tx + g.tgx * (ty + g.tgy * tz)]);
    return t * g.T + brick_code(g.dim, x & (g.bx - 1), y & (g.by - 1), z & (g.bz - 1));
}

// ------------------------------------------------------- FP64 <-> FP32 pairs

// FP32 -> FP64 from the bits, on the integer pipes (exact, as the conversion
// instruction; FP32 denormals, which the FP32 arithmetic flushes, give zero).
__device__ __forceinline__ double f2d_bits(float x)
{
    const unsigned X = __float_as_uint(x);
    const unsigned e = (X >> 23) & 0xffu;
    const unsigned ed = e == 0xffu ? 0x7ffu : e + 896u;
    const unsigned hi = (X & 0x80000000u) | (e ? (ed << 20) | ((X >> 3) & 0xfffffu) : 0u);
    const unsigned lo = e ? X << 29 : 0u;
    return __hiloint2double((int)hi, (int)lo);
}

// u = hi + lo to about 47 bits, from the bits of u on the integer and FP32
// pipes: hi is u with its 29 low mantissa bits cut off (exactly an FP32
// value, same sign), lo the cut-off part, rest * 2^(e - 1075), rounded once to
// FP32 (its two 16-bit halves convert exactly through the 2^23 magic number).
// |u| < 2^-126 stages as 0; |u| >= 2^116 (never a displacement) takes the
// conversion instruction.
__device__ __forceinline__ void split_bits(double u, float &hi, float &lo)
{
    const unsigned H = (unsigned)__double2hiint(u), Lw = (unsigned)__double2loint(u);
    const unsigned sign = H & 0x80000000u;
    const int e = (int)((H >> 20) & 0x7ffu);
    const unsigned rest = Lw & 0x1fffffffu;
    const float r1 = __uint_as_float(0x4b000000u | (rest >> 16)) - 8388608.f;
    const float r0 = __uint_as_float(0x4b000000u | (rest & 0xffffu)) - 8388608.f;
    const float fr = fmaf(r1, 65536.f, r0);
    // 2^(e - 1075) as 2^(e - 1011) * 2^-64, both normal FP32 numbers for 897 <= e <= 1138
    const float s1 = __uint_as_float((unsigned)(e - 884) << 23);
    const float l = fr * s1 * 5.42101086242752217e-20f;
    if (e < 897) {
        hi = 0.f;
        lo = 0.f;
    } else if (e > 1138) {
        hi = __double2float_rn(u);
        lo = 0.f;
    } else {
        hi = __uint_as_float(sign | ((unsigned)(e - 896) << 23) | ((H & 0xfffffu) << 3) | (Lw >> 29));
        lo = sign ? -l : l;
    }
}

// ------------------------------------------------------------ kernel args

// Row-wise passes of 3D lattices (pd_rows.cuh): the table holds 2 float4 per stencil
// entry, then one per segment and one of zeros.
constexpr int ROWS_PTAB = 280;      // float4 that fit the kernel parameter: m <= 3 (122 entries, 32 segments)
constexpr int ROWS_PLANES = 20;     // pair planes of the box: 4 + 2m, m <= 8
// The rules of the dispatch count tiles per SM of a GB300.
constexpr int SMS = 152;
// Grids of several waves of tiles: there the stencil tables go into the kernel parameter.
constexpr int PTAB_MIN_TILES = 2048;
// Where the row-wise passes take over (us a step, word-wise and row-wise):
// - PMB and the dilatation from two tiles per SM on (40^3 PMB, 125 tiles: 20.1 and 24.7; 64^3,
//   512 tiles: 49.2 and 46.6). Below, the word-wise kernels have twice as many threads per
//   tile.
// - PMB at m = 3 (128^3 277 and 247; summed in two ranges 329 and 261). Shorter horizons leave
//   segments of one and two bonds (m = 1: 128^3 96.3 and 110; m = 2: 80 x 80 x 72 32.3 and 33.9,
//   128^3 131 and 139), and at longer ones the word-wise kernel runs two threads a pair (m = 4:
//   64^3 88.6 and 99.5; m = 5: 169 and 176).
// - but not from 4.5 to 5 tiles per SM: the four CTAs of an SM end together here, so that the
//   last tiles gather on a few SMs (693 tiles 60.2 and 59.6, 704 to 756 60.2 and 65, 768 69.2
//   and 66.1).
// - the dilatation from m = 2 on (m = 1, LPS steps with the row-wise force: 56^3 25.2 and 26.9,
//   128^3 185 and 196).
// - the LPS force pass, at 128 registers and two CTAs per SM, from more than one tile per SM
//   on (45 x 37 x 52, 210 tiles: 36.9 and 34.2; 33 x 45 x 27 with m = 4, 120 tiles: 38.9 and 42.7),
//   where two CTAs' boxes fit in an SM (m = 5, one CTA: steps of 48^3 210 and 227, 56^3 292 and
//   313).
constexpr int ROWS_MIN_TILES = 2 * SMS, ROWS_MIN_TILES_FRC = SMS + 1;
inline bool rows_pmb(const Geom &g)
{
    return g.m == 3 && g.ntiles >= ROWS_MIN_TILES && !(2 * g.ntiles > 9 * SMS && g.ntiles <= 5 * SMS);
}
inline bool rows_dil(const Geom &g) { return g.m >= 2 && g.ntiles >= ROWS_MIN_TILES; }
inline bool rows_frc(const Geom &g, size_t smem)
{
    return g.ntiles >= ROWS_MIN_TILES_FRC && 2 * (smem + 1024) <= 228 * 1024;
}
struct RowArgs {
    const float4 *tab, *htab;       // device table and its host copy
    int ntab, nseg;                 // float4 of the table, segments
    int parts, split;               // ranges of stencil words summed apart (1 or 2); first segment of the second
    int nbox;                       // box entries
    int plane[ROWS_PLANES];         // entry of plane z' at column (-m, -m): its first rows are not stored
};

// Stencil entry of the all-FP64 passes (pd_f64.cu), in global memory (its warp-uniform
// reads hit the L1 while the FP64 pipe is busy).
struct F64Ent {
    double dx, dy, dz, d2;  // 2 d (PMB, LPS) or d (NP / LP); |d|^2
    double R, C, I;         // PMB: r0 / V_ij, r0^2 / V_ij, V_ij / r0; LPS: r0, V_ij; NP / LP: k, a'
    int off;                // box offset (x extent bx + 2m, y extent by + 2m)
    int near;               // PMB with s_c: high word of the num below which a bond is far from breaking
};

// One POD argument block for every tile kernel.
struct TileArgs {
    Geom g;
    const int4 *tile_org;
    const int *tile_ref;
    const int *tile_lut;
    const int4 *stencil;        // runtime stencil (dx, dy, dz, |d|^2) for generic kernels
    const double *stencil_r0;   // |d| of each stencil entry
    const float4 *src_hl;       // staging source (FP32C hi/lo pairs)
    const double4_32a *src_d4;      // staging source (FP64)
    float4 *dst_hl;             // next staging buffer written by MODE_STEP
    double4_32a *dst_d4;
    uint32_t *mask;
    double *u[3];
    double *v[3];
    const uint8_t *bc_kind;
    const double *bc_val;
    const double *body;
    double *f[3];               // MODE_FORCE output
    const float *minv32;        // LPS 1/m~
    const double *mtil;         // LPS m~ (FP64)
    float *theta32;
    double *theta64;
    double psi_beta;            // NP / LP potential rate
    const double *w[3];         // tangent input (slot order)
    double *jv[3];              // tangent output
    double *epoint;             // per-point energy (slot order)
    float4 *vhl;                // FP32C velocity as double-float pairs (2 float4 per slot)
    const float *bc32;          // FP32C boundary values as (hi, lo) per DOF, component-major
    const float4 *body32;       // FP32C body force per slot
    const float4 *tab_a;        // FP32C stencil table of the PMB and NP kernels (4 or NP_TAB_WORDS float4 / entry),
                                // or of the LPS dilatation (3 float4 / entry)
    const float4 *tab_b;        // FP32C stencil table of the LPS force pass (3 float4 / entry)
    const int *tile_nbr;        // [ntiles * 27] the 3^d neighbour tiles of each tile (or -1)
    int nbr_ok;                 // halo within one tile in every direction: tile_nbr is usable
    const uint32_t *box_map;    // paired halo box: neighbour tile (5 bits) + brick code (9) of A, then of B
    int box_edge[3];            // box_map holds for tiles with org <= box_edge on every axis
    float kF, kB;               // FP32C kick factors: dt/2 * fscale / rho and dt/2 / rho
    float dt_h, dt_l;           // dt as a double-float pair
    double fscale;              // force density = fscale * F (PMB: c V; LPS: 1/h)
    double cV;                  // c V (PMB)
    double inv_rho, dt, s_c, inv_h, h;
    double A, B;                // LPS 3K - 5 mu and 15 mu
    double K;                   // LPS bulk modulus (energy)
    int model;                  // PD_MODEL_PMB or PD_MODEL_LPS
    int v_is_half, update_breaking, mode, vol_corr, use_body, adjoint;
    int cd;                     // MODE_STEP: central-difference drift from u^{k-1} at dst
    int split;                  // fused bond kernels: threads per point pair (1, 2 or 4)
    int state64;                // FP32C fused update: u, v in the FP64 arrays u[], v[] (else double-float pairs)
    // host copies of tab_a / tab_b (read by the host launchers only: tables of at
    // most PTAB_N float4 are passed to the kernels as a parameter, see ParamTab)
    const float4 *htab_a, *htab_b;
    int ntab_a, ntab_b;
    const F64Ent *tab64;        // stencil table of the all-FP64 passes
    const RowArgs *rows;        // host: [2] the row-wise passes of this simulation (LPS dilatation; PMB, LPS force), or null
};

// A stencil table passed as a kernel parameter: the kernel reads it from the
// constant bank, whose warp-uniform reads take none of the shared-memory
// bandwidth that bounds the bond loops (128^3 LPS force pass 0.392 -> 0.361 ms
// against the same table in shared memory). 8 KB: 3D stencils up to m = 3.
constexpr int PTAB_N = 512;
struct ParamTab {
    float4 e[PTAB_N];
};

// --------------------------------------------------------------- staging

struct Ref32 { float hx, hy, hz, lx, ly, lz; };

__device__ __forceinline__ Ref32 tile_ref32(const TileArgs &a, int tile)
{
    int rs = __ldg(&a.tile_ref[tile]);
    float4 hi = __ldg(&a.src_hl[2 * rs]);
    float4 lo = __ldg(&a.src_hl[2 * rs + 1]);
    return Ref32{hi.x, hi.y, hi.z, lo.x, lo.y, lo.z};
}

__device__ __forceinline__ double3 tile_ref64(const TileArgs &a, int tile)
{
    int rs = __ldg(&a.tile_ref[tile]);
    double4_32a d = a.src_d4[rs];
    return make_double3(d.x, d.y, d.z);
}

// Fill the halo box (dims HX x HY x HZ, m-wide halo around the brick at org)
// with staged displacements in lattice units; points outside the grid get 0.
__device__ __forceinline__ void stage_box32(float4 *box, int HX, int HY, int nbox, int m,
                                            const TileArgs &a, const int4 &org, const Ref32 &ref,
                                            float inv_h)
{
    for (int b = threadIdx.x; b < nbox; b += blockDim.x) {
        int bxl = b % HX, rest = b / HX;
        int byl = rest % HY, bzl = rest / HY;
        int x = org.x + bxl - m, y = org.y + byl - m;
        int z = a.g.dim == 3 ? org.z + bzl - m : 0;
        int s = slot_at(a.g, a.tile_lut, x, y, z);
        float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s >= 0) {
            float4 hi = __ldg(&a.src_hl[2 * s]);
            float4 lo = __ldg(&a.src_hl[2 * s + 1]);
            r.x = ((hi.x - ref.hx) + (lo.x - ref.lx)) * inv_h;
            r.y = ((hi.y - ref.hy) + (lo.y - ref.ly)) * inv_h;
            r.z = ((hi.z - ref.hz) + (lo.z - ref.lz)) * inv_h;
        }
        box[b] = r;
    }
}

__device__ __forceinline__ void stage_box64(double4_32a *box, int HX, int HY, int nbox, int m,
                                            const TileArgs &a, const int4 &org, const double3 &ref,
                                            double inv_h)
{
    for (int b = threadIdx.x; b < nbox; b += blockDim.x) {
        int bxl = b % HX, rest = b / HX;
        int byl = rest % HY, bzl = rest / HY;
        int x = org.x + bxl - m, y = org.y + byl - m;
        int z = a.g.dim == 3 ? org.z + bzl - m : 0;
        int s = slot_at(a.g, a.tile_lut, x, y, z);
        double4_32a r = make_double4_32a(0.0, 0.0, 0.0, 0.0);
        if (s >= 0) {
            double4_32a d = a.src_d4[s];
            r.x = (d.x - ref.x) * inv_h;
            r.y = (d.y - ref.y) * inv_h;
            r.z = (d.z - ref.z) * inv_h;
        }
        box[b] = r;
    }
}

// ------------------------------------------------------------- epilogue

// Integrator update of one point from its internal force density f (N/m^3):
// MODE_STEP   v <- v + (dt or dt/2) a, then drift u <- u + dt v with boundary
//             conditions, and write the next staging buffer;
// MODE_FINALIZE  v <- v + dt/2 a (completes a half step), no drift;
// MODE_FORCE  store f.
// a = (f + b) / rho. Eqs. (7)-(9): the second half-kick of step k-1 and the
// first half-kick of step k use the same force f^k and run in the same kernel.
// With a.cd set a free DOF drifts by the central difference of Eq. (10),
// u^{k+1} = 2 u^k - u^{k-1} + dt^2 a^k, u^{k-1} read from the staging buffer
// the step overwrites.
__device__ __forceinline__ void point_epilogue(const TileArgs &a, int slot, const double f[3],
                                               int dim, bool fp64)
{
    const int ns = a.g.nslots;
    if (a.mode == MODE_FORCE) {
        for (int c = 0; c < dim; ++c) a.f[c][slot] = f[c];
        return;
    }
    double un[3] = {0.0, 0.0, 0.0};
    for (int c = 0; c < dim; ++c) {
        double acc = f[c];
        if (a.use_body) acc += a.body[c * ns + slot];
        acc *= a.inv_rho;
        double v = a.v[c][slot];
        const int kind = a.bc_kind[c * ns + slot];
        if (a.mode == MODE_STEP) {
            // second half-kick of the previous step (Eq. (9)), then the first
            // half-kick of this one (Eq. (7)), as two roundings like the equations
            const double hk = 0.5 * a.dt;
            if (a.v_is_half) v = fma(hk, acc, v);
            v = fma(hk, acc, v);
            double u = a.u[c][slot];
            if (kind == PD_BC_VELOCITY) {
                v = a.bc_val[c * ns + slot];
                u = fma(a.dt, v, u);
            } else if (kind == PD_BC_DISPLACEMENT) {
                v = 0.0;
                u = a.bc_val[c * ns + slot];
            } else if (a.cd) {
                double up;
                if (fp64) {
                    const double4_32a p = a.dst_d4[slot];
                    up = c == 0 ? p.x : (c == 1 ? p.y : p.z);
                } else {
                    const float4 ph = a.dst_hl[2 * slot], pl = a.dst_hl[2 * slot + 1];
                    up = c == 0 ? (double)ph.x + pl.x : (c == 1 ? (double)ph.y + pl.y : (double)ph.z + pl.z);
                }
                u = fma(a.dt * a.dt, acc, 2.0 * u - up);
            } else {
                u = fma(a.dt, v, u);
            }
            a.u[c][slot] = u;
            un[c] = u;
        } else {
            if (a.v_is_half) v = fma(0.5 * a.dt, acc, v);
            if (kind == PD_BC_VELOCITY) v = a.bc_val[c * ns + slot];
            else if (kind == PD_BC_DISPLACEMENT) v = 0.0;
        }
        a.v[c][slot] = v;
    }
    if (a.mode == MODE_STEP) {
        if (fp64) {
            a.dst_d4[slot] = make_double4_32a(un[0], un[1], un[2], 0.0);
        } else {
            float hx = (float)un[0], hy = (float)un[1], hz = (float)un[2];
            a.dst_hl[2 * slot] = make_float4(hx, hy, hz, 0.f);
            a.dst_hl[2 * slot + 1] = make_float4((float)(un[0] - (double)hx), (float)(un[1] - (double)hy),
                                                 (float)(un[2] - (double)hz), 0.f);
        }
    }
}

}  // namespace pdk
