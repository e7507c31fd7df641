// pd_krylov_grid.cu -- a GMRES cycle of pd_krylov.cu in one cooperative launch, for the
// cached tangent without a preconditioner: one block of 1024 threads per SM, a barrier
// over the grid where the other form ends a kernel.
//
// What bounds it. An Arnoldi step on the 200^2 plate (80,000 unknowns, 25 basis vectors on
// average) needs about 32 us of FP64 instructions (an SM issues one warp instruction every
// 16.6 cycles: the tangent product 15, the four passes over the basis 17) and took 107 us in
// ten kernels of a captured graph: short kernels that each start on an empty machine, wait
// on memory with one or two blocks per SM and end in a tail, one of them a single block (the
// Givens step, 11 us). Here every block owns a slice of the unknowns, so that an update and
// the products after it need no barrier between them; the step has seven barriers of 2 us.
// The sums count as much as the products: with a sum over the blocks done by every block for
// itself the step took 147 us (72 us of it FP64 additions), so each dot is summed by one warp
// of the grid. The last block owns no slice: it runs the Givens step while the others apply
// the tangent for the next one. Now 70 us: tangent 24, dots 14, updates 10, barriers and
// waits 14, sums and norm 8; 30^2 59 -> 39, 400^2 279 -> 192, 800^2 918 -> 627, the 200^2
// plate with an FP32 tangent 96 -> 66. Gathering several entries' loads before their products
// measured 74 (64 registers a thread: spills).
#include "pd_krylov.cuh"

namespace pdk {

constexpr int GT = 1024;                  // threads per block
constexpr int GW = GT / 32;
constexpr int GDOT = 512, GNORM = 128;    // elements of a slice per warp of a product, of a norm
constexpr int GSEG = 8;                   // warps per product at most

// ------------------------------------------------------------ grid barrier

// Every block of the cooperative launch arrives; bounded: a block that has waited
// wait_ns sets the word's top bit and returns false, and so does every block that finds
// it set (the count stays below it: 256 blocks at most, 7 arrivals a step, 500 steps).
constexpr unsigned GRID_FAILED = 0x80000000u;

__device__ __forceinline__ bool grid_barrier(unsigned *sync, unsigned &target, long long wait_ns)
{
    __shared__ int s_ok;
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned v;
        long long t0 = 0, t;
        asm volatile("atom.add.release.gpu.global.u32 %0, [%1], 1;" : "=r"(v) : "l"(sync) : "memory");
        for (unsigned polls = 0;; ++polls) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(sync) : "memory");
            if (v >= target) break;
            if (polls % 64) continue;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (polls == 0) t0 = t;
            if (t - t0 > wait_ns) {
                v = atomicOr(sync, GRID_FAILED) | GRID_FAILED;
                break;
            }
        }
        s_ok = v < GRID_FAILED;
    }
    __syncthreads();
    return s_ok != 0;
}

// Data that another block wrote in this launch is read through L2.

// y = A w of tangent_apply for the groups of 32 slots of block me of own: the 8 warps of a
// quarter of the block take every 8th stencil entry, their sums added in warp order.
template <class R, int DIM>
__device__ __forceinline__ void apply_groups(const TanOp &t, const double *w, double *y, int me, int own)
{
    __shared__ R part[GW / 8][2][7][DIM][32];   // sub 0 keeps its own
    const int quarter = threadIdx.x / 256, sub = threadIdx.x / 32 % 8, lane = threadIdx.x % 32;
    const size_t ns = t.nslots;
    const R *coef = static_cast<const R *>(t.coef);
    constexpr int NC = DIM == 3 ? 6 : 3;
    const int groups = (t.nslots + 31) / 32;
    int buf = 0;
    for (int g = me + quarter * own; g < groups; g += GW / 8 * own, buf ^= 1) {   // each SM within one group of the others
        const int s = 32 * g + lane;
        const bool act = s < t.nslots && __ldg(&t.user_of_slot[s]) >= 0;
        R a0 = 0, a1 = 0, a2 = 0;
        if (act) {
            const double wi0 = __ldcg(&w[s]), wi1 = __ldcg(&w[ns + s]), wi2 = DIM == 3 ? __ldcg(&w[2 * ns + s]) : 0.0;
#pragma unroll 4
            for (int k = sub; k < t.S; k += 8) {
                const int j = __ldg(&t.nbr[(size_t)k * ns + s]);
                const R *D = coef + (size_t)k * NC * ns + s;
                const R d0 = (R)(__ldcg(&w[j]) - wi0), d1 = (R)(__ldcg(&w[ns + j]) - wi1);
                const R xx = __ldg(&D[0]), xy = __ldg(&D[ns]), yy = __ldg(&D[2 * ns]);
                if (DIM == 3) {
                    const R d2 = (R)(__ldcg(&w[2 * ns + j]) - wi2);
                    const R xz = __ldg(&D[3 * ns]), yz = __ldg(&D[4 * ns]), zz = __ldg(&D[5 * ns]);
                    a0 += xx * d0 + xy * d1 + xz * d2;
                    a1 += xy * d0 + yy * d1 + yz * d2;
                    a2 += xz * d0 + yz * d1 + zz * d2;
                } else {
                    a0 += xx * d0 + xy * d1;
                    a1 += xy * d0 + yy * d1;
                }
            }
        }
        auto &p = part[quarter][buf];
        if (sub > 0) {
            p[sub - 1][0][lane] = a0;
            p[sub - 1][1][lane] = a1;
            if (DIM == 3) p[sub - 1][DIM - 1][lane] = a2;
        }
        asm volatile("bar.sync %0, 256;" ::"r"(1 + quarter) : "memory");
        if (sub == 0 && s < t.nslots) {
#pragma unroll
            for (int c = 0; c < DIM; ++c) {
                const size_t e = (size_t)c * ns + s;
                if (!act) {
                    y[e] = 0.0;
                    continue;
                }
                R acc = c == 0 ? a0 : c == 1 ? a1 : a2;
#pragma unroll
                for (int q = 0; q < 7; ++q) acc += p[q][c][lane];
                y[e] = __ldg(&t.kind[e]) == PD_BC_DISPLACEMENT ? __ldcg(&w[e]) : -(double)acc;
            }
        }
    }
}

// partial[i ldp] = V_i . w over the slice [lo, hi) for i < k: nseg warps a vector, their
// sums (buf, k nseg) added in order.
__device__ __forceinline__ void slice_dots(const double *V, int k, const double *w, long long n, long long lo, long long hi,
                                           int nseg, double *buf, double *partial, int ldp)
{
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const long long seg = ((hi - lo + nseg - 1) / nseg + 31) / 32 * 32;
    __syncthreads();   // the slice of w is complete, buf is free
    for (int u = warp; u < k * nseg; u += GW) {
        const double *vi = V + (long long)(u / nseg) * n;
        const long long a = lo + (u % nseg) * seg, b = min(hi, a + seg);
        double acc = 0.0;
#pragma unroll 8
        for (long long e = a + lane; e < b; e += 32) acc = fma(__ldcg(&vi[e]), __ldcg(&w[e]), acc);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) buf[u] = acc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < k; i += GT) {
        double acc = buf[i * nseg];
        for (int q = 1; q < nseg; ++q) acc += buf[i * nseg + q];
        partial[(long long)i * ldp] = acc;
    }
}

// The sum of nb slices' partials, by one warp (every lane has it).
__device__ __forceinline__ double slices_total(const double *p, int nb)
{
    double acc = 0.0;
    for (int b = threadIdx.x % 32; b < nb; b += 32) acc += __ldcg(&p[b]);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

// Arnoldi steps 0 .. steps - 1 of a cycle (V_0 and the scalars are set). V_0 stays as it is,
// so that a cycle whose wait ran out can be run again. stall (tests): block 0 does not take
// part, so that the others' first wait runs out.
template <class R, int DIM>
__global__ void __launch_bounds__(GT, 1) k_gmres_grid(const __grid_constant__ TanOp t, double *V, long long n,
                                                     double *partial, double *d, int m, int steps, unsigned *sync,
                                                     long long wait_ns, int stall)
{
    if (stall && blockIdx.x == 0) return;
    extern __shared__ double sm[];          // h (m + 1), the products' sums; the last block: 3 (m + 1)
    double *h = sm, *buf = sm + m + 1;
    __shared__ double s_norm2, s_inv;
    const GmLayout L(m);
    const int own = gridDim.x - 1, me = blockIdx.x, warp = threadIdx.x / 32;
    const bool last = me == own;
    const long long per = ((n + own - 1) / own + 31) / 32 * 32;
    const long long lo = min(n, me * per), hi = last ? lo : min(n, lo + per);
    const int nseg = (int)min((long long)GSEG, max(1LL, per / GDOT)), nnorm = (int)min((long long)GW, max(1LL, per / GNORM));
    unsigned target = 0;
    for (int j = 0; j < steps; ++j) {
        double *w = V + (long long)(j + 1) * n;
        if (!last) apply_groups<R, DIM>(t, V + (long long)j * n, w, me, own);
        else if (j > 0) gm_givens(d, m, j - 1, s_norm2, buf);
        if (!grid_barrier(sync, target, wait_ns)) return;
        if (j > 0 && __ldcg(&d[L.sc + GM_DONE]) != 0.0) return;
        for (int pass = 0; pass < 2; ++pass) {
            if (!last) slice_dots(V, j + 1, w, n, lo, hi, nseg, buf, partial + me, own);
            if (!grid_barrier(sync, target, wait_ns)) return;
            if (warp == 0)
                for (int i = me; i <= j; i += own + 1) {
                    const double x = slices_total(partial + (long long)i * own, own);
                    if (threadIdx.x == 0) {
                        double *H = d + L.H + i + (m + 1) * j;
                        d[i] = x;
                        *H = pass ? *H + x : x;
                    }
                }
            if (!grid_barrier(sync, target, wait_ns)) return;
            for (int i = threadIdx.x; i <= j; i += GT) h[i] = __ldcg(&d[i]);
            __syncthreads();
            for (long long e = lo + threadIdx.x; e < hi; e += GT) {
                double acc = __ldcg(&w[e]);
#pragma unroll 8
                for (int i = 0; i <= j; ++i) acc = fma(-h[i], __ldcg(&V[(long long)i * n + e]), acc);
                w[e] = acc;
            }
        }
        if (!last) slice_dots(w, 1, w, n, lo, hi, nnorm, buf, partial + me, own);
        if (!grid_barrier(sync, target, wait_ns)) return;
        if (warp == 0) {
            const double x = slices_total(partial, own);
            if (threadIdx.x == 0) {    // one thread: a square root and a quotient by every warp took 5 us
                const double hn = sqrt(x);
                s_norm2 = x;
                s_inv = hn > 0.0 ? 1.0 / hn : 0.0;
            }
        }
        __syncthreads();
        const double inv = s_inv;
        for (long long e = lo + threadIdx.x; e < hi; e += GT) w[e] = inv * __ldcg(&w[e]);
        if (!grid_barrier(sync, target, wait_ns)) return;
    }
    if (last) gm_givens(d, m, steps - 1, s_norm2, buf);
}

// ------------------------------------------------------------------- launch

template <class F>
static int go(F *k, int smem, void **args, unsigned *sync, cudaStream_t st)
{
    int dev = 0, sms = 0, ctas = 0;
    PD_CUDA(cudaGetDevice(&dev));
    PD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (smem > 160 * 1024 || cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024) != cudaSuccess) {
        cudaGetLastError();
        return PD_ENOTREADY;
    }
    PD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, k, GT, smem));
    if (ctas < 1 || sms < 2) return PD_ENOTREADY;
    PD_CUDA(cudaMemsetAsync(sync, 0, sizeof(unsigned), st));
    const cudaError_t e = cudaLaunchCooperativeKernel(k, dim3(std::min(sms, GRID_MAX)), dim3(GT), args, smem, st);
    if (e == cudaSuccess) return PD_OK;
    cudaGetLastError();
    return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported ? PD_ENOTREADY
                                                                                 : cuda_fail(e, "cooperative launch");
}

int gmres_grid(const TanOp &t, double *V, long long n, double *partial, double *d, int m, int steps, long long wait_ns,
               int stall, cudaStream_t st)
{
    unsigned *sync = reinterpret_cast<unsigned *>(d + GmLayout(m).size());
    void *args[] = {(void *)&t, &V, &n, &partial, &d, &m, &steps, &sync, &wait_ns, &stall};
    const int smem = (m + 1 + std::max(GSEG * (m + 1), GW)) * (int)sizeof(double);
    if (t.fp64) return go(t.dim == 3 ? k_gmres_grid<double, 3> : k_gmres_grid<double, 2>, smem, args, sync, st);
    return go(t.dim == 3 ? k_gmres_grid<float, 3> : k_gmres_grid<float, 2>, smem, args, sync, st);
}

}  // namespace pdk
