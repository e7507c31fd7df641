// pd_lists.cu -- the neighbour build on lattices whose halo stays within one tile
// (Sec. 3.1; Sec. 4.2.1): the bond masks and their sums by class of points, and the CSR
// rows by tile. Every output equals the cell-list build's (pd_build.cu), which the wider
// horizons keep.
//
// The horizon of a point is the stencil clipped to the grid, so its bond mask, its number
// of bonds and the sums over them (weighted volume, stable step) depend only on its
// distances to the six faces, each counted up to m: at most (2m + 1)^3 classes. One thread
// per class evaluates them, in the stencil order of k_stencil_sum, and a pass over the
// slots copies its class's values (64^3, m = 3: 381 us of counting and summing kernels -> 21).
//
// A row of the CSR is the point's neighbours in ascending Morton rank, which is (tile
// number, code within the tile). The points of a tile's halo box fall into its 27
// neighbour tiles; within one they are the same codes for every tile, so their position
// in the box's rank order is (the points of the neighbour tiles with smaller numbers) +
// (a fixed index in the own one). A warp per row sets its neighbours' positions as bits;
// a neighbour's place in the row is then the number of set bits below its own (a prefix
// over the words and one popcount): no sort, no candidate test, and the row leaves in
// coalesced stores (64^3: 590 -> 163 us, writing 121 MB; reading the set bits back in order,
// each lane storing its own, took 349). It is bound by the shared-memory pipe (83 %).
#include <stdlib.h>

#include <algorithm>

#include "pd_tile.cuh"

namespace pdk {

int exclusive_scan(const int *in, long long n, long long *out, cudaStream_t st);

// Classes per axis: every coordinate on short axes, else those less than m from either
// face and one for the rest. Class -> a coordinate of it, coordinate -> class.
__host__ __device__ inline int axis_classes(int n, int m) { return n < 2 * m + 1 ? n : 2 * m + 1; }
__device__ __forceinline__ int axis_coord(int c, int n, int m) { return c <= m || n <= 2 * m + 1 ? c : n - (2 * m + 1) + c; }
__device__ __forceinline__ int axis_class(int x, int n, int m)
{
    if (n <= 2 * m + 1 || x <= m) return x;
    return x >= n - m ? x - (n - (2 * m + 1)) : m;
}

// Per class: mask words, number of bonds, and the two sums of k_stencil_sum.
__global__ void __launch_bounds__(64) k_class(Geom g, int vol_corr, int kx, int ky, int kz, const int4 *stencil,
                                              const double *stencil_r0, uint32_t *cmask, int *ccount, double *csum_m,
                                              unsigned long long *smax)
{
    // the entries' values by all threads, so that a class's loop is left with the additions
    extern __shared__ double ctab[];
    double *tm = ctab, *td = ctab + g.S;
    int4 *sd = reinterpret_cast<int4 *>(ctab + 2 * ((g.S + 1) & ~1));
    for (int k = threadIdx.x; k < g.S; k += blockDim.x) {
        const double r0 = __ldg(&stencil_r0[k]);
        const double v = vol_corr ? vol_factor_lattice(g.m, r0) : 1.0;
        sd[k] = __ldg(&stencil[k]);
        tm[k] = __dmul_rn((double)sd[k].w, v);
        td[k] = v / r0;
    }
    __syncthreads();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= kx * ky * kz) return;
    const int x = axis_coord(c % kx, g.nx, g.m), y = axis_coord((c / kx) % ky, g.ny, g.m),
              z = axis_coord(c / (kx * ky), g.nz, g.m);
    int count = 0;
    double am = 0.0, ad = 0.0;
    for (int w = 0; w < g.W; ++w) {
        uint32_t word = 0u;
        const int nb = min(32, g.S - 32 * w);
        for (int b = 0; b < nb; ++b) {
            const int4 d = sd[32 * w + b];
            if ((unsigned)(x + d.x) >= (unsigned)g.nx || (unsigned)(y + d.y) >= (unsigned)g.ny ||
                (unsigned)(z + d.z) >= (unsigned)g.nz)
                continue;
            word |= 1u << b;
            ++count;
            am = __dadd_rn(am, tm[32 * w + b]);
            ad = __dadd_rn(ad, td[32 * w + b]);
        }
        cmask[(size_t)c * g.W + w] = word;
    }
    ccount[c] = count;
    csum_m[c] = am;
    // positive doubles order like their bit patterns; every class has points
    atomicMax(smax, (unsigned long long)__double_as_longlong(ad));
}

// Per slot: its class's mask words, row length and (LPS) weighted volume.
__global__ void __launch_bounds__(256) k_class_apply(Geom g, int kx, int ky, const int4 *tile_org,
                                                     const int *rank_of_slot, const uint32_t *cmask, const int *ccount,
                                                     const double *csum_m, uint32_t *mask, int *row_count, double *mtil,
                                                     float *minv32)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.nslots) return;
    const int4 o = __ldg(&tile_org[s >> g.L]);
    int l[3];
    morton_decode(g.dim, (uint64_t)(s & (g.T - 1)), l);
    const int x = o.x + l[0], y = o.y + l[1], z = o.z + l[2];
    const bool in = x < g.nx && y < g.ny && z < g.nz;
    const int c = in ? axis_class(x, g.nx, g.m) + kx * (axis_class(y, g.ny, g.m) + ky * axis_class(z, g.nz, g.m)) : 0;
    for (int w = 0; w < g.W; ++w) mask[(size_t)w * g.nslots + s] = in ? __ldg(&cmask[(size_t)c * g.W + w]) : 0u;
    if (!in) return;
    row_count[rank_of_slot[s]] = __ldg(&ccount[c]);
    if (mtil) {
        const double acc = __ldg(&csum_m[c]);
        mtil[s] = acc;
        minv32[s] = acc > 0.0 ? (float)(1.0 / acc) : 0.f;
    }
}

constexpr int LIST_WARPS = 8;

// One CTA per tile. box_tab: per entry of the halo box its neighbour tile (27), its code
// and its index among the box's points of that tile; box_cnt: the box's points per
// neighbour tile.
__global__ void __launch_bounds__(32 * LIST_WARPS) k_tile_rows(Geom g, const int4 *tile_org, const int *tile_nbr,
                                                               const uint32_t *box_tab, const int *box_cnt, int nbox,
                                                               const int4 *stencil, const int *rank_of_slot,
                                                               const uint32_t *mask, int stage_mask, const int64_t *row_ptr, int *col)
{
    extern __shared__ int lsm[];
    const int nw = (nbox + 31) / 32;
    int *rk = lsm;                                              // Morton rank by position
    int *off = rk + nbox;                                       // box offset of each stencil entry
    int *rows = off + g.S;                                      // per warp, the row
    uint32_t *bits = reinterpret_cast<uint32_t *>(rows + LIST_WARPS * g.S);     // per warp, one bit per position
    uint16_t *below = reinterpret_cast<uint16_t *>(bits + LIST_WARPS * nw);     // per warp, set bits before each word
    uint16_t *pos = below + LIST_WARPS * nw;
    // the rows' starts and mask words, loaded together (one row at a time, each warp waited
    // for three loads in turn: 309 us)
    __shared__ long long s_start[512];
    __shared__ uint16_t s_own[512];
    uint32_t *smask = reinterpret_cast<uint32_t *>(pos + ((nbox + 1) & ~1));
    __shared__ int s_nbr[27], s_base[27];
    const int tile = blockIdx.x, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int HX = g.bx + 2 * g.m, HY = g.by + 2 * g.m;
    if (threadIdx.x < 27) s_nbr[threadIdx.x] = __ldg(&tile_nbr[27 * tile + threadIdx.x]);
    for (int k = threadIdx.x; k < g.S; k += blockDim.x) {
        const int4 d = __ldg(&stencil[k]);
        off[k] = d.x + HX * (d.y + HY * d.z);
    }
    for (int k = threadIdx.x; k < LIST_WARPS * nw; k += blockDim.x) bits[k] = 0u;
    __syncthreads();
    if (threadIdx.x < 27) {
        // points of the neighbour tiles with smaller numbers (absent ones, -1, hold none)
        int b = 0;
        const int t = s_nbr[threadIdx.x];
        for (int k = 0; k < 27; ++k)
            if (s_nbr[k] >= 0 && s_nbr[k] < t) b += __ldg(&box_cnt[k]);
        s_base[threadIdx.x] = t >= 0 ? b : -1;
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nbox; b += blockDim.x) {
        const uint32_t e = __ldg(&box_tab[b]);
        const int k = e & 31u;
        int p = 0;
        if (s_base[k] >= 0) {
            p = s_base[k] + (int)(e >> 14);
            rk[p] = __ldg(&rank_of_slot[s_nbr[k] * g.T + (int)((e >> 5) & 511u)]);
        }
        pos[b] = (uint16_t)p;
    }
    for (int t = threadIdx.x; t < g.T; t += blockDim.x) {
        const int r = __ldg(&rank_of_slot[tile * g.T + t]);
        s_start[t] = r >= 0 ? row_ptr[r] : -1;
        int l[3];
        morton_decode(g.dim, (uint64_t)t, l);
        s_own[t] = (uint16_t)((l[0] + g.m) + HX * ((l[1] + g.m) + HY * (g.dim == 3 ? l[2] + g.m : 0)));
        if (stage_mask)
            for (int w = 0; w < g.W; ++w) smask[w * g.T + t] = __ldg(&mask[(size_t)w * g.nslots + tile * g.T + t]);
    }
    __syncthreads();
    uint32_t *my = bits + warp * nw;
    uint16_t *pre = below + warp * nw;
    int *row = rows + warp * g.S;
    // gridDim.y CTAs share a tile's rows on grids of few tiles
    for (int t = warp + LIST_WARPS * blockIdx.y; t < g.T; t += LIST_WARPS * gridDim.y) {
        const long long base = s_start[t];
        if (base < 0) continue;                                 // off the lattice
        const uint32_t *mk = stage_mask ? smask + t : mask + tile * g.T + t;
        const size_t mw = stage_mask ? g.T : g.nslots;
        const uint16_t *po = pos + s_own[t];
        // the lane's neighbours k = lane + 32 i: the first four positions stay in registers
        int p4[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            p4[i] = -1;
            if (i < g.W && ((mk[i * mw] >> lane) & 1u)) {
                p4[i] = po[off[32 * i + lane]];
                atomicOr(&my[p4[i] >> 5], 1u << (p4[i] & 31));
            }
        }
        for (int i = 4; i < g.W; ++i)
            if ((mk[i * mw] >> lane) & 1u) {
                const int p = po[off[32 * i + lane]];
                atomicOr(&my[p >> 5], 1u << (p & 31));
            }
        __syncwarp();
        int total = 0;
        for (int w0 = 0; w0 < nw; w0 += 32) {
            const int n = w0 + lane < nw ? __popc(my[w0 + lane]) : 0;
            int at = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, at, o);
                if (lane >= o) at += v;
            }
            if (w0 + lane < nw) pre[w0 + lane] = (uint16_t)(total + at - n);
            total += __shfl_sync(0xffffffffu, at, 31);
        }
        __syncwarp();
        auto put = [&](int p) { row[pre[p >> 5] + __popc(my[p >> 5] & ((1u << (p & 31)) - 1u))] = rk[p]; };
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (p4[i] >= 0) put(p4[i]);
        for (int i = 4; i < g.W; ++i)
            if ((mk[i * mw] >> lane) & 1u) put(po[off[32 * i + lane]]);
        __syncwarp();
        for (int w = lane; w < nw; w += 32) my[w] = 0u;
        for (int k = lane; k < total; k += 32) col[base + k] = row[k];
        __syncwarp();
    }
}

size_t tile_rows_smem(const Geom &g, int nbox)
{
    const size_t nw = (nbox + 31) / 32;
    return sizeof(int) * ((size_t)nbox + g.S + LIST_WARPS * ((size_t)g.S + nw)) +
           sizeof(uint16_t) * (LIST_WARPS * nw + (((size_t)nbox + 1) & ~(size_t)1));
}

// Masks, weighted volume, max_i sum_j V_ij / |d| (d_sum_max) and the CSR. Stream-ordered:
// the number of bonds is the offsets' count on the lattice, nothing is read back.
int build_tile_lists(const Geom &g, const Material &mat, const Tables &t, const int4 *host_stencil, const int *tile_nbr,
                     const uint32_t *box_tab, const int *box_cnt, int nbox, BuildOut *out, uint32_t *mask, double *mtil,
                     float *minv32, double *d_sum_max, cudaStream_t st)
{
    const long long n = g.npoints;
    const int kx = axis_classes(g.nx, g.m), ky = axis_classes(g.ny, g.m), kz = axis_classes(g.nz, g.m), nc = kx * ky * kz;
    out->row_ptr = nullptr;
    out->col = nullptr;
    out->nbonds = 0;
    for (int k = 0; k < g.S; ++k) {
        const int4 d = host_stencil[k];
        const long long a = g.nx - abs(d.x), b = g.ny - abs(d.y), c = g.nz - abs(d.z);
        if (a > 0 && b > 0 && c > 0) out->nbonds += a * b * c;
    }
    // scratch: csum_m, row_count, ccount, cmask
    const size_t bytes = sizeof(double) * nc + sizeof(int) * (size_t)n + sizeof(int) * nc + sizeof(uint32_t) * (size_t)nc * g.W;
    char *buf = nullptr;
    // the mask words too where they leave room for several CTAs per SM
    const int stage_mask = (size_t)g.W * g.T <= 4096;
    const size_t smem = tile_rows_smem(g, nbox) + (stage_mask ? sizeof(uint32_t) * (size_t)g.W * g.T : 0);
    if (lib_malloc(reinterpret_cast<void **>(&buf), bytes, st) != cudaSuccess ||
        lib_malloc(reinterpret_cast<void **>(&out->row_ptr), sizeof(int64_t) * (n + 1), st) != cudaSuccess ||
        lib_malloc(reinterpret_cast<void **>(&out->col), sizeof(int) * std::max(1LL, (long long)out->nbonds), st) != cudaSuccess) {
        cudaGetLastError();
        lib_free(buf, st);
        lib_free(out->row_ptr, st);
        lib_free(out->col, st);
        out->row_ptr = nullptr;
        out->col = nullptr;
        set_error("device allocation of the neighbour lists (%lld bonds) failed", (long long)out->nbonds);
        return PD_ENOMEM;
    }
    double *csum = reinterpret_cast<double *>(buf);
    int *row_count = reinterpret_cast<int *>(csum + nc), *ccount = row_count + n;
    uint32_t *cmask = reinterpret_cast<uint32_t *>(ccount + nc);
    cudaMemsetAsync(d_sum_max, 0, sizeof(double), st);
    k_class<<<(nc + 63) / 64, 64, (2 * sizeof(double) + sizeof(int4)) * (g.S + 1), st>>>(g, mat.vol_corr, kx, ky, kz, t.stencil, t.stencil_r0, cmask, ccount, csum,
                                           reinterpret_cast<unsigned long long *>(d_sum_max));
    k_class_apply<<<(g.nslots + 255) / 256, 256, 0, st>>>(g, kx, ky, t.tile_org, t.rank_of_slot, cmask, ccount, csum, mask,
                                                          row_count, mtil, minv32);
    int rc = exclusive_scan(row_count, n, reinterpret_cast<long long *>(out->row_ptr), st);
    cudaError_t e = smem_limit(k_tile_rows, smem);
    if (rc == PD_OK && e == cudaSuccess) {
        k_tile_rows<<<dim3(g.ntiles, std::min(8, std::max(1, 4 * SMS / g.ntiles))), 32 * LIST_WARPS, smem, st>>>(g, t.tile_org, tile_nbr, box_tab, box_cnt, nbox, t.stencil,
                                                             t.rank_of_slot, mask, stage_mask, out->row_ptr, out->col);
        e = cudaGetLastError();
    }
    lib_free(buf, st);
    if (rc == PD_OK && e != cudaSuccess) rc = cuda_fail(e, "neighbour lists");
    return rc;
}

}  // namespace pdk
