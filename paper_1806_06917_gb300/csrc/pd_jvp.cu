// pd_jvp.cu -- tangent Jacobian-vector product of the PMB internal force and its
// adjoint: the matrix-free replacement of the central-difference stiffness
// assembly of Eq. (6) / Algorithm 3.
//
// With f_pair(eta) = c s n, n = y/|y|, s = (|y| - |xi|)/|xi| and y = xi + eta,
//   d f_pair / d eta = c [ n n^T / |xi| + s (I - n n^T) / |y| ] =: D_ij,
//   (K w)_i = sum_j D_ij (w_j - w_i) V_j V_ij.
// In lattice units (|xi| = h|d|, |y| = h r):
//   (K w)_i = (c V / h) sum_j V_ij [ (n.dw)(1/|d| - s/r) n + (s/r) dw ].
// The adjoint is the transposed gather
//   (K^T v)_i = sum_j D_ji V_i V_ij v_j - sum_j D_ij V_j V_ij v_i
// with D_ji computed here, in FP32, from the bond as seen from j (xi -> -xi, eta -> -eta).
// The volumes are uniform and D_ji = D_ij, so the FP64 product (pd_f64.cu) serves both.
// Displacements are staged as in the force kernels; the direction w is staged
// relative to the tile's reference value so that w_j - w_i keeps its precision.
#include "pd_tile.cuh"

namespace pdk {

int launch_f64_jvp(const TileArgs &a, size_t smem, cudaStream_t st);

__global__ void __launch_bounds__(256) jvp_fp32(const TileArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Geom &g = a.g;
    const int m = g.m;
    const int HX = g.bx + 2 * m, HY = g.by + 2 * m, HZ = g.dim == 3 ? g.bz + 2 * m : 1;
    const int nbox = HX * HY * HZ;
    float4 *box = reinterpret_cast<float4 *>(smem_raw);
    float4 *wbox = box + nbox;
    const int tile = blockIdx.x;
    const int4 org = __ldg(&a.tile_org[tile]);
    stage_box32(box, HX, HY, nbox, m, a, org, tile_ref32(a, tile), (float)a.inv_h);
    const int rs_slot = __ldg(&a.tile_ref[tile]);
    const double wr[3] = {a.w[0][rs_slot], a.w[1][rs_slot], g.dim == 3 ? a.w[2][rs_slot] : 0.0};
    for (int b = threadIdx.x; b < nbox; b += blockDim.x) {
        int x, y, z;
        box_coord(b, HX, HY, m, g.dim, org, x, y, z);
        const int s = slot_at(g, a.tile_lut, x, y, z);
        float4 r;
        r.x = r.y = r.z = r.w = 0.f;
        if (s >= 0) {
            r.x = (float)(a.w[0][s] - wr[0]);
            r.y = (float)(a.w[1][s] - wr[1]);
            if (g.dim == 3) r.z = (float)(a.w[2][s] - wr[2]);
        }
        wbox[b] = r;
    }
    __syncthreads();

    const int adj = a.adjoint;
    for (int t = threadIdx.x; t < g.T; t += blockDim.x) {
        const int lx = t % g.bx, ly = (t / g.bx) % g.by, lz = t / (g.bx * g.by);
        const int slot = tile * g.T + brick_code(g.dim, lx, ly, lz);
        if (!(org.x + lx < g.nx && org.y + ly < g.ny && org.z + lz < g.nz)) continue;
        const int bi = (lx + m) + HX * ((ly + m) + HY * (g.dim == 3 ? lz + m : 0));
        const float4 ui = box[bi];
        const float4 wi = wbox[bi];
        float ox = 0, oy = 0, oz = 0;
        for (int w = 0; w < g.W; ++w) {
            const uint32_t word = a.mask[(size_t)w * g.nslots + slot];
            const int nb = min(32, g.S - 32 * w);
            for (int b = 0; b < nb; ++b) {
                if (!((word >> b) & 1u)) continue;
                const int4 d = __ldg(&a.stencil[32 * w + b]);
                const float r0 = (float)__ldg(&a.stencil_r0[32 * w + b]);
                const int bj = bi + d.x + HX * (d.y + HY * d.z);
                const float4 uj = box[bj];
                const float4 wj = wbox[bj];
                // bond geometry from i's side, or from j's side for the adjoint
                const float sg = adj ? -1.f : 1.f;
                const float ex = sg * (uj.x - ui.x), ey = sg * (uj.y - ui.y), ez = sg * (uj.z - ui.z);
                const float dx = sg * (float)d.x, dy = sg * (float)d.y, dz = sg * (float)d.z;
                const float yx = ex + dx, yy = ey + dy, yz = ez + dz;
                const float q = yx * yx + yy * yy + yz * yz;
                const float num = ex * ex + ey * ey + ez * ez + 2.f * (dx * ex + dy * ey + dz * ez);
                const float rs = prsqrt1(q);
                const float s = pdiv1(num, r0 * (q * rs + r0));
                // D (w_j - w_i); volumes are uniform, so V_i / V_j placement is 1
                const float dwx = wj.x - wi.x, dwy = wj.y - wi.y, dwz = wj.z - wi.z;
                const float ndw = (yx * dwx + yy * dwy + yz * dwz) * rs;
                const float cn = ndw * (1.f / r0 - s * rs) * rs;
                const float cs = s * rs;
                const float vij = a.vol_corr ? (float)vol_factor_lattice(m, (double)r0) : 1.f;
                ox += vij * (cn * yx + cs * dwx);
                oy += vij * (cn * yy + cs * dwy);
                oz += vij * (cn * yz + cs * dwz);
            }
        }
        const double sc = a.cV * a.inv_h;
        a.jv[0][slot] = sc * (double)ox;
        a.jv[1][slot] = sc * (double)oy;
        if (g.dim == 3) a.jv[2][slot] = sc * (double)oz;
    }
}

size_t jvp_smem(const Geom &g, int precision)
{
    const size_t nbox = (size_t)(g.bx + 2 * g.m) * (g.by + 2 * g.m) * (g.dim == 3 ? g.bz + 2 * g.m : 1);
    return 2 * nbox * (precision == PD_FP64 ? sizeof(double4_32a) : sizeof(float4));
}

int launch_jvp_args(const TileArgs &a, int precision, cudaStream_t st)
{
    const size_t smem = jvp_smem(a.g, precision);
    if (precision == PD_FP64) return launch_f64_jvp(a, smem, st);
    PD_CUDA(smem_limit(jvp_fp32, smem));
    jvp_fp32<<<a.g.ntiles, 256, smem, st>>>(a);
    PD_CUDA(cudaGetLastError());
    return PD_OK;
}

}  // namespace pdk
