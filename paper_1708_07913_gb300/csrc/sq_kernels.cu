// sq_kernels.cu -- setup and FP64 post-processing kernels of libsq:
//   * potential copy with a periodic halo (Section 3.1 periodic index map)
//   * separable Gaussian projector tables (KB projectors restricted to the
//     region of influence, Section 3.1)
//   * extreme eigenvalues of the Lanczos tridiagonals (Section 3.2)
//   * quadrature weights by discrete orthogonality (Eq. cqj)
//   * Fermi level by a bracketing search on the electron count (Section 3.2)
//   * density, band energy and entropy (Eqs. ElectronDensity, Eband, Entropy)
// Every global sum is deterministic: per-block tree sums in a fixed order,
// then the last block to finish adds the block partials in index order.
#include <math.h>
#include <algorithm>
#include "sq_internal.cuh"

namespace sq {

// ------------------------------------------------------------------------
// Potential with halo: Vp[k'][j'][i'] = V[(k'-m) mod n3][(j'-m) mod n2][(i'-m) mod n1]
// ------------------------------------------------------------------------
template <typename T>
__global__ void vpad_kernel(const double* __restrict__ V, T* __restrict__ Vp, int n1, int n2, int n3, int m,
                            unsigned* err)
{
    const long long tot = (long long)(n1 + 2 * m) * (n2 + 2 * m) * (n3 + 2 * m);
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x)
        vpad_elem<T>(V, Vp, n1, n2, n3, m, t, err);
}

int launch_build_vpad(sq_ctx* ctx, const double* V)
{
    const GridParams& g = ctx->g;
    long long tot = (long long)g.P1 * g.P2 * (g.n3 + 2 * g.m);
    int blocks = (int)std::min<long long>((tot + 255) / 256, (long long)ctx->sm_count * 16);
    if (ctx->precision == SQ_FP32)
        vpad_kernel<float><<<blocks, 256, 0, ctx->stream>>>(V, (float*)ctx->Vp, g.n1, g.n2, g.n3, g.m, ctx->d_err);
    else
        vpad_kernel<double><<<blocks, 256, 0, ctx->stream>>>(V, (double*)ctx->Vp, g.n1, g.n2, g.n3, g.m, ctx->d_err);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

// ------------------------------------------------------------------------
// Projector tables.  For atom I at R with box start lo (atom-relative grid
// index) the displacement along axis a of box point i is d = (lo_a + i) h - R_a
// (rounded multiply then subtract, no FMA, so the support test below matches a
// plain evaluation of the same expression).  G = exp(-d^2/(2 rc^2)), DG = d G.
// Row (jj,kk) keeps the x-range of points with d_x^2 + d_y^2 + d_z^2 < r_nl^2.
// ------------------------------------------------------------------------
template <typename T>
__global__ void proj_table_kernel(const double* __restrict__ R, const AtomTab* __restrict__ at, int n_atoms,
                                  int lb, double h, double rc, double rnl2, T* G, T* DG, uint8_t* ivl)
{
    const int atom = blockIdx.x;
    if (atom >= n_atoms) return;
    const AtomTab A = at[atom];
    const double two_rc2 = 2.0 * rc * rc;
    for (int t = threadIdx.x; t < 3 * lb; t += blockDim.x) {
        int ax = t / lb, i = t % lb;
        double g = 0.0, dg = 0.0;
        if (i < A.len[ax]) {
            double d = __dadd_rn(__dmul_rn((double)(A.lo[ax] + i), h), -R[3 * atom + ax]);
            g = exp(-__dmul_rn(d, d) / two_rc2);
            dg = d * g;
        }
        G[((size_t)atom * 3 + ax) * lb + i] = (T)g;
        DG[((size_t)atom * 3 + ax) * lb + i] = (T)dg;
    }
    for (int t = threadIdx.x; t < lb * lb; t += blockDim.x) {
        int jj = t / lb, kk = t % lb;
        int xlo = 1, xhi = 0;
        if (jj < A.len[1] && kk < A.len[2]) {
            double dy = __dadd_rn(__dmul_rn((double)(A.lo[1] + jj), h), -R[3 * atom + 1]);
            double dz = __dadd_rn(__dmul_rn((double)(A.lo[2] + kk), h), -R[3 * atom + 2]);
            int first = -1, last = -1;
            for (int ii = 0; ii < A.len[0]; ++ii) {
                double dx = __dadd_rn(__dmul_rn((double)(A.lo[0] + ii), h), -R[3 * atom + 0]);
                double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                if (r2 < rnl2) {
                    if (first < 0) first = ii;
                    last = ii;
                }
            }
            if (first >= 0) { xlo = first; xhi = last; }
        }
        ivl[(((size_t)atom * lb + jj) * lb + kk) * 2 + 0] = (uint8_t)xlo;
        ivl[(((size_t)atom * lb + jj) * lb + kk) * 2 + 1] = (uint8_t)xhi;
    }
}

int launch_proj_tables(sq_ctx* ctx, const double* d_R)
{
    double rnl2 = ctx->rnl * ctx->rnl;
    if (ctx->precision == SQ_FP32)
        proj_table_kernel<float><<<ctx->n_atoms, 256, 0, ctx->stream>>>(
            d_R, ctx->d_atoms, ctx->n_atoms, ctx->lb, ctx->g.h, ctx->rc, rnl2, (float*)ctx->d_G, (float*)ctx->d_DG,
            ctx->d_ivl);
    else
        proj_table_kernel<double><<<ctx->n_atoms, 256, 0, ctx->stream>>>(
            d_R, ctx->d_atoms, ctx->n_atoms, ctx->lb, ctx->g.h, ctx->rc, rnl2, (double*)ctx->d_G, (double*)ctx->d_DG,
            ctx->d_ivl);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

// Support rows as 32-bit column masks, [atom][plane kk][row jj] (boxes have at
// most NL_BOX = 32 columns): what the quad kernels cut their lists from.
__global__ void support_mask_kernel(const uint8_t* __restrict__ ivl, int n_atoms, int lb, uint32_t* __restrict__ mask)
{
    const long long n = (long long)n_atoms * lb * lb;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int jj = (int)(t % lb), kk = (int)((t / lb) % lb);
        const long long atom = t / ((long long)lb * lb);
        const uchar2 iv = *reinterpret_cast<const uchar2*>(ivl + ((atom * lb + jj) * lb + kk) * 2);
        mask[t] = iv.x <= iv.y ? (0xffffffffu >> (31 - iv.y)) & (0xffffffffu << iv.x) : 0u;
    }
}

// The most projector entries of any region row.  Every row of a node's region is
// the middle row of some node's (periodic grid), so each node counts that one.
__global__ void row_entries_kernel(const AtomTab* __restrict__ at, const uint8_t* __restrict__ ivl,
                                   const int* __restrict__ tile_start, const int4* __restrict__ tile_cand, int nt0,
                                   int nt1, int lb, int n1, int n2, long long Nd, int m, int* most)
{
    int best = 0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < Nd; q += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(q % n1), j = (int)((q / n1) % n2), k = (int)(q / ((long long)n1 * n2));
        const int tile = i / TILE + nt0 * (j / TILE + nt1 * (k / TILE));
        int n = 0;
        for (int c = tile_start[tile]; c < tile_start[tile + 1]; ++c) {
            const int4 tc = tile_cand[c];
            const int jj = j - tc.z, kk = k - tc.w;
            if (jj < 0 || kk < 0 || jj >= at[tc.x].len[1] || kk >= at[tc.x].len[2]) continue;
            const uchar2 iv = *reinterpret_cast<const uchar2*>(ivl + (((size_t)tc.x * lb + jj) * lb + kk) * 2);
            n += iv.x <= iv.y && tc.y + iv.y >= i - m && tc.y + iv.x <= i + m;
        }
        best = max(best, n);
    }
    best = __reduce_max_sync(0xffffffffu, (unsigned)best);
    if ((threadIdx.x & 31) == 0) atomicMax(most, best);
}

// The quad kernels' support masks (ctx->d_qmask, one more word for the result of
// the second kernel) and the most entries of any region row.  Waits.
int launch_support_masks(sq_ctx* ctx, int* most_row_entries)
{
    const long long n = (long long)ctx->n_atoms * ctx->lb * ctx->lb;
    int* most = reinterpret_cast<int*>(ctx->d_qmask + n);
    support_mask_kernel<<<(int)std::min<long long>((n + 255) / 256, (long long)ctx->sm_count * 8), 256, 0, ctx->stream>>>(
        ctx->d_ivl, ctx->n_atoms, ctx->lb, ctx->d_qmask);
    SQ_CUDA_TRY(cudaMemsetAsync(most, 0, sizeof(int), ctx->stream));
    row_entries_kernel<<<(int)std::min<long long>((ctx->g.Nd + 127) / 128, (long long)ctx->sm_count * 16), 128, 0,
                         ctx->stream>>>(ctx->d_atoms, ctx->d_ivl, ctx->d_tile_start, ctx->d_tile_cand, ctx->ntile[0],
                                        ctx->ntile[1], ctx->lb, ctx->g.n1, ctx->g.n2, ctx->g.Nd, ctx->g.m, most);
    ctx->launches += 2;
    SQ_CUDA_TRY(cudaMemcpyAsync(most_row_entries, most, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    SQ_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

// ------------------------------------------------------------------------
// Extreme eigenvalues of the Lanczos tridiagonal T_k by Sturm bisection.
// The count of eigenvalues below x is the number of sign changes of the
// leading principal minors p_0 = 1, p_i = (a_i - x) p_{i-1} - b_{i-1}^2 p_{i-2}
// (an exact zero takes the sign opposite to its predecessor).  Minors are
// rescaled by powers of two to stay in range; no division is needed.
//
// FP64 bounds it (two lanes per clock and SM), so signs and exponents are read
// from the high words and a step is left with three FP64 operations; a node has
// two threads, one per end of the spectrum, in blocks of one warp, which also
// spreads small grids over the SMs, and its coefficients (b squared) lie in
// shared memory.
// ------------------------------------------------------------------------
constexpr int TRI_NODES = 16;                     // nodes of a block (one warp)

__device__ inline int hi_word(double v) { return __double2hiint(v); }

// Eigenvalues below x; a and b2 with stride TRI_NODES.
__device__ int sturm_count(int k, const double* a, const double* b2, double x)
{
    double pm = 1.0, p = 1.0, bb = 0.0;
    int cnt = 0;
    unsigned sprev = 0;                           // sign bit of the predecessor
    for (int i = 0; i < k; ++i) {
        const double pn = (a[i * TRI_NODES] - x) * p - bb * pm;
        pm = p;
        p = pn;
        bb = b2[i * TRI_NODES];
        const int h = hi_word(p), m = hi_word(pm);
        const bool zero = ((h & 0x7fffffff) | __double2loint(p)) == 0;
        const unsigned s = zero ? sprev ^ 1u : (unsigned)h >> 31;
        cnt += s != sprev;
        sprev = s;
        const int eh = h & 0x7fffffff, em = m & 0x7fffffff;
        constexpr int BIG = (1023 + 256) << 20, SMALL = (1023 - 256) << 20;
        if (eh > BIG || em > BIG) { p *= 0x1p-256; pm *= 0x1p-256; }
        else if (eh < SMALL && em < SMALL) { p *= 0x1p+256; pm *= 0x1p+256; }
    }
    return cnt;
}

// One warp per TRI_NODES nodes: lane = node + 16 * end (0: smallest, 1: largest eigenvalue).
__global__ void __launch_bounds__(32) tridiag_bounds_kernel(const double* __restrict__ alpha, const double* __restrict__ beta,
                                                            const int* __restrict__ klen, int cap, int steps,
                                                            long long Nd, double margin, double* __restrict__ chi,
                                                            double* __restrict__ zeta)
{
    extern __shared__ double tsm[];               // a then b^2, [steps][TRI_NODES] each
    const int lane = threadIdx.x, n = lane & (TRI_NODES - 1), end = lane >> 4;
    double* A = tsm + n;
    double* B = tsm + (size_t)steps * TRI_NODES + n;
    for (long long q0 = (long long)blockIdx.x * TRI_NODES; q0 < Nd; q0 += (long long)gridDim.x * TRI_NODES) {
        const long long q = q0 + n < Nd ? q0 + n : Nd - 1;
        const int k = min(klen[q], steps);
        const double* a = alpha + q * cap;
        const double* b = beta + q * cap;
        __syncwarp();
        double glo = INFINITY, ghi = -INFINITY;
        for (int i = 0; i < k; ++i) {
            const double r = (i > 0 ? fabs(b[i - 1]) : 0.0) + (i < k - 1 ? fabs(b[i]) : 0.0);
            glo = fmin(glo, a[i] - r);
            ghi = fmax(ghi, a[i] + r);
            if (end == 0) A[i * TRI_NODES] = a[i];
            else B[i * TRI_NODES] = i < k - 1 ? b[i] * b[i] : 0.0;
        }
        __syncwarp();
        const double pad = 1e-12 * (fabs(glo) + fabs(ghi)) + 1e-300;
        double lo = glo - pad, hi = ghi + pad;
        const int want = end == 0 ? 1 : k;
        for (int it = 0; it < 200; ++it) {
            const double mid = 0.5 * (lo + hi);
            if (mid == lo || mid == hi) break;
            if (sturm_count(k, A, B, mid) >= want) hi = mid; else lo = mid;
        }
        __syncwarp();
        const double theta = 0.5 * (lo + hi), other = __shfl_xor_sync(0xffffffffu, theta, TRI_NODES);
        if (end == 0 && q0 + n < Nd) {
            const double tmin = theta, tmax = other;
            const double width = fmax(tmax - tmin, 1.0);
            const double L = tmin - margin * width, H = tmax + margin * width;
            chi[q] = 0.5 * (H + L);
            zeta[q] = 0.5 * (H - L);
        }
    }
}

// Extremes of the tridiagonals of n_lanczos steps (the rows of alpha and beta hold ctx->nl_cap); shared memory for
// these steps only: 48 x 49 x 50 regions of 5^3, 40 steps, take 36.7 ms, and 57.3 with the rows' 512 in shared memory.
int launch_tridiag_bounds(sq_ctx* ctx, int n_lanczos, double margin, double* chi, double* zeta)
{
    const long long Nd = ctx->g.Nd;
    const int blocks = (int)std::min<long long>((Nd + TRI_NODES - 1) / TRI_NODES, (long long)ctx->sm_count * 32);
    const size_t bytes = (size_t)2 * n_lanczos * TRI_NODES * sizeof(double);        // at most 512 steps: 128 KB
    if (bytes > 48 * 1024) {                      // raise only (see the region kernels' dispatch)
        cudaFuncAttributes fa;
        if (cudaFuncGetAttributes(&fa, tridiag_bounds_kernel) != cudaSuccess) return SQ_ECUDA;
        if ((int)bytes > fa.maxDynamicSharedSizeBytes &&
            cudaFuncSetAttribute(tridiag_bounds_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) !=
                cudaSuccess)
            return SQ_ECUDA;
    }
    tridiag_bounds_kernel<<<blocks, 32, bytes, ctx->stream>>>(ctx->d_alpha, ctx->d_beta, ctx->d_klen, ctx->nl_cap,
                                                              n_lanczos, Nd, margin, chi, zeta);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

// ------------------------------------------------------------------------
// Quadrature weights (Eq. cqj by discrete orthogonality at the zeros x_k of
// T_{npl+1}):  W_qk = (2/K) [ rho^0/2 + sum_{j>=1} rho^j T_j(x_k) ],  K = npl+1,
// stored zero by zero ([K][Nd]) so that the kernels with a thread per node read
// them coalesced.  T_j(x_{K-1-k}) = (-1)^j T_j(x_k): the even and the odd part
// of the sum serve two zeros, which halves the FP64 multiply-adds that bound
// the kernel (two lanes per clock and SM).  A block takes 32 nodes, a lane each,
// and its warps the zeros; T_j(x_k) from a table in shared memory, or by the three-term
// recurrence where K x K/2 doubles do not fit.
// ------------------------------------------------------------------------
constexpr int WT_NODES = 32, WT_T = 256;

__global__ void __launch_bounds__(WT_T) weights_kernel(const double* __restrict__ mom, double* __restrict__ W, long long Nd,
                                                       int K, int use_table)
{
    extern __shared__ double wsm[];
    const int H = (K + 1) / 2, KP = K | 1;               // odd pitch: lanes in distinct banks
    double* r = wsm;                                     // [WT_NODES][KP] moments, rho^0 halved
    double* T = wsm + WT_NODES * KP;                     // [H][K]: T_j(x_k)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (use_table)
        for (int k = threadIdx.x; k < H; k += WT_T) {
            const double x = cos(M_PI * (k + 0.5) / K);
            double tm = 1.0, t = x;
            T[k * K] = 1.0;
            T[k * K + 1] = x;
            for (int j = 2; j < K; ++j) {
                const double tn = 2.0 * x * t - tm;
                tm = t;
                t = tn;
                T[k * K + j] = t;
            }
        }
    const double c = 2.0 / K;
    for (long long q0 = (long long)blockIdx.x * WT_NODES; q0 < Nd; q0 += (long long)gridDim.x * WT_NODES) {
        const int nq = (int)(Nd - q0 < WT_NODES ? Nd - q0 : WT_NODES);
        __syncthreads();
        for (int i = threadIdx.x; i < nq * K; i += WT_T) {
            const int n = i / K, j = i - n * K;
            const double v = mom[q0 * K + i];
            r[n * KP + j] = j == 0 ? 0.5 * v : v;
        }
        __syncthreads();
        if (lane < nq) {
            const double* rn = r + lane * KP;
            for (int k = warp; k < H; k += WT_T / 32) {
                double e = rn[0], o = 0.0;
                if (use_table) {
                    const double* Tk = T + k * K;
                    int j = 1;
                    for (; j + 1 < K; j += 2) {
                        o += rn[j] * Tk[j];
                        e += rn[j + 1] * Tk[j + 1];
                    }
                    if (j < K) o += rn[j] * Tk[j];
                } else {
                    const double x = cos(M_PI * (k + 0.5) / K);
                    double tm = 1.0, t = x;
                    for (int j = 1; j < K; ++j) {
                        if (j & 1) o += rn[j] * t;
                        else e += rn[j] * t;
                        const double tn = 2.0 * x * t - tm;
                        tm = t;
                        t = tn;
                    }
                }
                W[(long long)k * Nd + q0 + lane] = c * (e + o);
                if (K - 1 - k != k) W[(long long)(K - 1 - k) * Nd + q0 + lane] = c * (e - o);
            }
        }
    }
}

int launch_weights(sq_ctx* ctx, const double* moments)
{
    const int K = ctx->npl + 1, H = (K + 1) / 2;
    const size_t rows = (size_t)WT_NODES * (K | 1) * sizeof(double), table = (size_t)H * K * sizeof(double);
    const int use_table = rows + table <= 100 * 1024;
    const size_t bytes = rows + (use_table ? table : 0);
    if (bytes > 48 * 1024) {                      // raise only (see the region kernels' dispatch)
        cudaFuncAttributes fa;
        if (cudaFuncGetAttributes(&fa, weights_kernel) != cudaSuccess) return SQ_ECUDA;
        if ((int)bytes > fa.maxDynamicSharedSizeBytes &&
            cudaFuncSetAttribute(weights_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess)
            return SQ_ECUDA;
    }
    const int blocks = (int)std::min<long long>((ctx->g.Nd + WT_NODES - 1) / WT_NODES, (long long)ctx->sm_count * 4);
    weights_kernel<<<blocks, WT_T, bytes, ctx->stream>>>(moments, ctx->d_W, ctx->g.Nd, K, use_table);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

// ------------------------------------------------------------------------
// Deterministic grid reductions (last-block-done pattern).
// ------------------------------------------------------------------------
constexpr int RED_T = 256;

__device__ inline double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum NV doubles over the block; result valid in thread 0.
template <int NV>
__device__ inline void block_reduce(double (&v)[NV], double* sh)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = warp_sum_d(v[i]);
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < NV; ++i) sh[i * 32 + w] = v[i];
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            double t = 0.0;
            for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += sh[i * 32 + k];
            v[i] = t;
        }
    }
}

// Fermi state (doubles): the first FERMI_STATE are read by the host.
enum { F_LO = 0, F_HI, F_NE, F_KT, F_NLO, F_NHI, F_DONE, F_ITERS, F_STATUS, F_EB, F_ES, F_NEL, F_NSTATE,
       F_FINE = 12, F_NPTS, F_PTS };
constexpr int FERMI_PTS = 7;
constexpr int FERMI_MAX = 200;                            // passes of a search, at most
static_assert(F_NSTATE == FERMI_STATE && F_PTS + FERMI_PTS <= 32, "Fermi state size");

// Sum of one value per thread over the partials of all blocks, by the whole of
// the last block in a fixed order; valid in thread 0.
template <int NV>
__device__ inline void sum_partials(const double* red, unsigned nb, double (&v)[NV], double* sh)
{
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        v[i] = 0.0;
        for (unsigned b = threadIdx.x; b < nb; b += blockDim.x) v[i] += __ldcg(red + (size_t)NV * b + i);
    }
    __syncthreads();
    block_reduce<NV>(v, sh);
}

// min(chi - zeta) - 10 kT and max(chi + zeta) + 10 kT; the ends are the first points of the search.
__global__ void fermi_bracket_kernel(const double* __restrict__ chi, const double* __restrict__ zeta, long long Nd,
                                     double* red, unsigned* count, double* st)
{
    __shared__ double sh[64];
    __shared__ bool last;
    double lo = INFINITY, hi = -INFINITY;
    auto block_minmax = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        if ((threadIdx.x & 31) == 0) { sh[threadIdx.x >> 5] = lo; sh[32 + (threadIdx.x >> 5)] = hi; }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int k = 0; k < (int)(blockDim.x >> 5); ++k) { lo = fmin(lo, sh[k]); hi = fmax(hi, sh[32 + k]); }
    };
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < Nd;
         q += (long long)gridDim.x * blockDim.x) {
        lo = fmin(lo, chi[q] - zeta[q]);
        hi = fmax(hi, chi[q] + zeta[q]);
    }
    block_minmax();
    if (threadIdx.x == 0) {
        red[2 * blockIdx.x] = lo;
        red[2 * blockIdx.x + 1] = hi;
        __threadfence();
        last = atomicAdd(count, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    lo = INFINITY;
    hi = -INFINITY;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
        lo = fmin(lo, __ldcg(red + 2 * b));
        hi = fmax(hi, __ldcg(red + 2 * b + 1));
    }
    __syncthreads();
    block_minmax();
    if (threadIdx.x == 0) {
        st[F_LO] = st[F_PTS] = lo - 10.0 * st[F_KT];
        st[F_HI] = st[F_PTS + 1] = hi + 10.0 * st[F_KT];
        st[F_NPTS] = 2.0;
        st[F_FINE] = -1.0;                                // the ends come first
        st[F_DONE] = 0.0;
        st[F_ITERS] = 0.0;
        st[F_STATUS] = 0.0;
        *count = 0;
    }
}

// First zero k with chi + zeta x_k - mu <= 41 kT, or up to two before it (x_k
// falls with k, FP32, the margin covers its rounding): where the terms begin
// that are not 0.  With the sign of the bound turned, past which they are 1.
// An interval run through backwards or of one point (z <= 0) has no such order:
// every zero is visited.
__device__ inline int zero_index(double c, double z, double bound, int K, bool up)
{
    const float zf = (float)z, x = fminf(1.0f, fmaxf(-1.0f, (float)(bound - c) / zf));
    const float k = acosf(x) * (float)K * 0.318309886f - 0.5f;
    const int i = up ? (int)ceilf(k) + 1 : (int)floorf(k) - 1;
    return zf > 0.0f ? min(K, max(0, i)) : up ? K : 0;
}

// The next points of the search (thread 0).  lo < hi bracket the electron
// count, fl and fh the counts there.
__device__ void fermi_next(double* st, double lo, double hi, double fl, double fh, int coarse)
{
    const double mid = 0.5 * (lo + hi), w = hi - lo, kT = st[F_KT];
    st[F_LO] = lo;
    st[F_HI] = hi;
    st[F_NLO] = fl;
    st[F_NHI] = fh;
    double p[FERMI_PTS];
    int n = 0;
    const double tiny = 8.0 * 2.220446049250313e-16 * fmax(fabs(lo), fabs(hi));
    if (mid == lo || mid == hi) {                         // adjacent in FP64
        st[F_DONE] = 1.0;
        return;
    }
    const bool fine = w < 0.25 * kT;
    if (!fine && coarse == 1) {
        p[n++] = mid;
    } else if (!fine || w <= 8.0 * tiny) {                // two or three levels of bisection at once
        const double a = 0.5 * (lo + mid), b = 0.5 * (mid + hi);
        if (fine) p[n++] = 0.5 * (lo + a);
        p[n++] = a;
        if (fine) p[n++] = 0.5 * (a + mid);
        p[n++] = mid;
        if (fine) p[n++] = 0.5 * (mid + b);
        p[n++] = b;
        if (fine) p[n++] = 0.5 * (b + hi);
    } else {                                              // the count is smooth on the scale kT: around the secant
        const double x = lo + w * ((st[F_NE] - fl) / (fh - fl));
        const double d = 0.25 * w * (w / kT) + 0.25 * tiny;
        const double off[6] = {-8.0 * d, -d, 0.0, d, 8.0 * d, mid - x};
        for (int i = 0; i < 6; ++i) {
            const double v = x + off[i];
            if (v > lo && v < hi) p[n++] = v;
        }
        if (n == 0) p[n++] = mid;
        for (int i = 1; i < n; ++i)                       // ascending
            for (int j = i; j > 0 && p[j] < p[j - 1]; --j) {
                const double t = p[j];
                p[j] = p[j - 1];
                p[j - 1] = t;
            }
    }
    for (int i = 0; i < n; ++i) st[F_PTS + i] = p[i];
    st[F_NPTS] = (double)n;
    st[F_FINE] = fine ? 1.0 : 0.0;
}

// The bracket that the counts acc at the points leave, and the next points (thread 0).
__device__ void fermi_decide(double* st, const double (&acc)[FERMI_PTS], const double* pts, int np, bool fine, int coarse)
{
    const double Ne = st[F_NE];
    if (st[F_FINE] < -0.5) {                              // the ends
        if (!(acc[0] <= Ne && acc[1] >= Ne)) {
            st[F_NLO] = acc[0];
            st[F_NHI] = acc[1];
            st[F_STATUS] = (double)SQ_ENOCONV;
            st[F_DONE] = 1.0;
            return;
        }
        fermi_next(st, st[F_LO], st[F_HI], acc[0], acc[1], coarse);
        return;
    }
    double lo = st[F_LO], hi = st[F_HI], fl = st[F_NLO], fh = st[F_NHI];
    // three points of one bisection tree (coarse) are walked as bisection walks them; else the first rise past Ne
    if (!fine && np == 3) {
        const int i = acc[1] < Ne ? 2 : 0;
        if (i == 2) { lo = pts[1]; fl = acc[1]; } else { hi = pts[1]; fh = acc[1]; }
        if (acc[i] < Ne) { lo = pts[i]; fl = acc[i]; } else { hi = pts[i]; fh = acc[i]; }
    } else {
        for (int i = 0; i < np; ++i) {
            if (acc[i] < Ne) {
                lo = pts[i];
                fl = acc[i];
            } else {
                hi = pts[i];
                fh = acc[i];
                break;
            }
        }
    }
    st[F_ITERS] += 1.0;
    fermi_next(st, lo, hi, fl, fh, coarse);
    if (st[F_ITERS] >= FERMI_MAX) st[F_DONE] = 1.0;
}

// Electron count N(mu) = 2 sum_q sum_k W_qk g((chi_q + zeta_q x_k - mu)/kT) at
// up to FERMI_PTS points at once, then (last block) the bracket they leave and
// the next points.  Beyond |t| = 40 the Fermi factor is 1.0 exactly in FP64
// (t < -40) or below 4.3e-18 (t > 40, dropped: < 1e-16 of any count here), so a
// node visits only the zeros around mu.  What bounds it is FP64 (two lanes per
// clock and SM): a term is an exponential and a division; within a bracket far
// narrower than kT the points share the exponential, e^{(E-mu)/kT} = a s.  The
// level, density and energies of 64^3 nodes at n_pl 48 took 31.8 ms with about
// 60 bisection passes that each visited every zero, one node's row per thread,
// and take 7.5 ms now.
template <bool MANY>
__global__ void fermi_search_kernel(const double* __restrict__ W, const double* __restrict__ chi,
                                    const double* __restrict__ zeta, long long Nd, int K, int coarse, int rounds,
                                    double* red, unsigned* count, double* st)
{
    __shared__ double sh[FERMI_PTS * 32];
    __shared__ bool last;
    __shared__ double xk[MAX_NPL + 1], pts[FERMI_PTS], sc[FERMI_PTS];
    if (st[F_DONE] != 0.0) return;                        // uniform over the grid
    for (int k = threadIdx.x; k < K; k += blockDim.x) xk[k] = cos(M_PI * (k + 0.5) / K);
    for (int round = 0; round < (MANY ? rounds : 1); ++round) {      // MANY: a grid of one block
        const double kT = st[F_KT];
        const int np = (int)st[F_NPTS];
        const bool fine = st[F_FINE] > 0.5;
        const double ref = st[F_PTS + (np >> 1)];
        if ((int)threadIdx.x < np) {
            pts[threadIdx.x] = st[F_PTS + threadIdx.x];
            sc[threadIdx.x] = fine ? exp((ref - st[F_PTS + threadIdx.x]) / kT) : 0.0;
        }
        __syncthreads();
        double acc[FERMI_PTS];
#pragma unroll
        for (int i = 0; i < FERMI_PTS; ++i) acc[i] = 0.0;
        for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < Nd;
             q += (long long)gridDim.x * blockDim.x) {
            const double c = chi[q], z = zeta[q];
            const double* w = W + q;
            if (fine) {
                const int ka = zero_index(c, z, pts[np - 1] + 41.0 * kT, K, false);
                const int kb = zero_index(c, z, pts[0] - 41.0 * kT, K, true);
                double s[FERMI_PTS], full = 0.0;
#pragma unroll
                for (int i = 0; i < FERMI_PTS; ++i) s[i] = 0.0;
                for (int k = ka; k < kb; ++k) {
                    const double wk = w[(long long)k * Nd], a = exp((c + z * xk[k] - ref) / kT);
#pragma unroll
                    for (int i = 0; i < FERMI_PTS; ++i)
                        if (i < np) s[i] += wk / (1.0 + a * sc[i]);
                }
                for (int k = max(ka, kb); k < K; ++k) full += w[(long long)k * Nd];
#pragma unroll
                for (int i = 0; i < FERMI_PTS; ++i)
                    if (i < np) acc[i] += 2.0 * (s[i] + full);
            } else {
#pragma unroll
                for (int i = 0; i < FERMI_PTS; ++i) {
                    if (i >= np) break;
                    const double mu = pts[i];
                    const int ka = zero_index(c, z, mu + 41.0 * kT, K, false);
                    const int kb = zero_index(c, z, mu - 41.0 * kT, K, true);
                    double s = 0.0;
                    for (int k = ka; k < kb; ++k) {
                        const double t = (c + z * xk[k] - mu) / kT;
                        if (t > 40.0) continue;
                        const double wk = w[(long long)k * Nd];
                        s += (t < -40.0) ? wk : wk / (1.0 + exp(t));
                    }
                    for (int k = max(ka, kb); k < K; ++k) s += w[(long long)k * Nd];
                    acc[i] += 2.0 * s;
                }
            }
        }
        block_reduce<FERMI_PTS>(acc, sh);
        if (threadIdx.x == 0) {
            for (int i = 0; i < FERMI_PTS; ++i) red[(size_t)FERMI_PTS * blockIdx.x + i] = acc[i];
            __threadfence();
            last = atomicAdd(count, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        sum_partials<FERMI_PTS>(red, gridDim.x, acc, sh);
        if (threadIdx.x == 0) {
            *count = 0;
            fermi_decide(st, acc, pts, np, fine, coarse);
        }
        if (!MANY) return;
        __syncthreads();
        if (st[F_DONE] != 0.0) return;
    }
}

// Search state reset (a kernel rather than a host copy, so the whole
// Fermi-level search can be captured in a CUDA graph).
__global__ void fermi_init_kernel(double* st, double Ne, double kT)
{
    if (threadIdx.x == 0) {
        for (int i = 0; i < F_NSTATE; ++i) st[i] = 0.0;
        st[F_NE] = Ne;
        st[F_KT] = kT;
    }
}

// Blocks of 256 threads where that fills the GPU, else of 64, so that small systems spread over the SMs.
static int node_threads(long long Nd, int sm_count) { return Nd >= (long long)sm_count * 512 ? RED_T : 64; }
static int node_blocks(const sq_ctx* ctx, int threads)
{
    return (int)std::min<long long>((ctx->g.Nd + threads - 1) / threads, ctx->red_blocks);
}

// Launches of one pass each over the whole GPU; one block that makes all the passes left.
static int enqueue_search(sq_ctx* ctx, const double* chi, const double* zeta, int launches, bool one_block = false)
{
    const int T = node_threads(ctx->g.Nd, ctx->sm_count), B = node_blocks(ctx, T);
    // far from the level a large system takes one point per pass (FP64-bound), a small one three (launch-bound)
    const int coarse = ctx->g.Nd >= 65536 ? 1 : 3;
    auto launch = [&](auto kernel, int blocks, int threads) {
        kernel<<<blocks, threads, 0, ctx->stream>>>(ctx->d_W, chi, zeta, ctx->g.Nd, ctx->npl + 1, coarse, FERMI_MAX,
                                                    ctx->d_red, ctx->d_count, ctx->d_fermi);
    };
    for (int it = 0; it < launches; ++it)
        if (one_block) launch(fermi_search_kernel<true>, 1, RED_T);
        else launch(fermi_search_kernel<false>, B, T);
    ctx->launches += launches;
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

static int enqueue_search_start(sq_ctx* ctx, const double* chi, const double* zeta, double Ne, double kT)
{
    const int T = node_threads(ctx->g.Nd, ctx->sm_count);
    fermi_init_kernel<<<1, 32, 0, ctx->stream>>>(ctx->d_fermi, Ne, kT);
    fermi_bracket_kernel<<<node_blocks(ctx, T), T, 0, ctx->stream>>>(chi, zeta, ctx->g.Nd, ctx->d_red, ctx->d_count,
                                                                     ctx->d_fermi);
    ctx->launches += 2;
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

// A pass at least halves the bracket, and the search ends when its midpoint equals
// an end point: after 53 + log2(spectrum / |mu|) halvings or so where the count is
// flat around mu, and after 20 to 45 passes otherwise.  Passes past the end return
// at once.  A caller that waits queues lots of FERMI_FIRST until the search says
// that it has ended; a captured search queues FERMI_PASSES, and the rest (hardly
// ever any) are made by one block, which needs no further launches.
constexpr int FERMI_PASSES = 56, FERMI_FIRST = 18;

// Enqueue the whole Fermi-level search on ctx->stream (no host wait); the
// result stays in the device state: mu = (st[F_LO] + st[F_HI]) / 2, status
// in st[F_STATUS].
int enqueue_fermi(sq_ctx* ctx, const double* chi, const double* zeta, double Ne, double kT)
{
    int rc = enqueue_search_start(ctx, chi, zeta, Ne, kT);
    if (rc || (rc = enqueue_search(ctx, chi, zeta, FERMI_PASSES))) return rc;
    return enqueue_search(ctx, chi, zeta, 1, true);
}

int run_fermi(sq_ctx* ctx, const double* chi, const double* zeta, double Ne, double kT, double* mu)
{
    int rc = enqueue_search_start(ctx, chi, zeta, Ne, kT);
    if (rc) return rc;
    double st[F_NSTATE];
    for (int done = 0; done <= FERMI_MAX; done += FERMI_FIRST) {              // most searches end in the first lot
        if ((rc = enqueue_search(ctx, chi, zeta, FERMI_FIRST))) return rc;
        SQ_CUDA_TRY(cudaMemcpyAsync(st, ctx->d_fermi, sizeof(st), cudaMemcpyDeviceToHost, ctx->stream));
        SQ_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
        if (st[F_DONE] != 0.0) break;
    }
    if (st[F_STATUS] != 0.0) return (int)st[F_STATUS];
    *mu = 0.5 * (st[F_LO] + st[F_HI]);
    return SQ_OK;
}

int fermi_result(const double* st_host, double* mu, double* eb, double* es, double* ne)
{
    if (mu) *mu = 0.5 * (st_host[F_LO] + st_host[F_HI]);
    if (eb) *eb = st_host[F_EB];
    if (es) *es = st_host[F_ES];
    if (ne) *ne = st_host[F_NEL];
    return st_host[F_STATUS] != 0.0 ? (int)st_host[F_STATUS] : SQ_OK;
}

// ------------------------------------------------------------------------
// Density, band energy, entropy, electron count at mu.
// ------------------------------------------------------------------------
__global__ void density_kernel(const double* __restrict__ W, const double* __restrict__ chi,
                               const double* __restrict__ zeta, long long Nd, int K, double mu, double kT, double h,
                               double* __restrict__ rho, double* red, unsigned* count, double* st, int mu_from_state)
{
    __shared__ double sh[96];
    __shared__ bool last;
    __shared__ double xk[MAX_NPL + 1];
    if (mu_from_state) mu = 0.5 * (((volatile double*)st)[F_LO] + ((volatile double*)st)[F_HI]);
    for (int k = threadIdx.x; k < K; k += blockDim.x) xk[k] = cos(M_PI * (k + 0.5) / K);
    __syncthreads();
    const double h3 = h * h * h;
    double acc[3] = {0.0, 0.0, 0.0};   // E_band, E_ent, N
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < Nd;
         q += (long long)gridDim.x * blockDim.x) {
        const double c = chi[q], z = zeta[q];
        const double* w = W + q;
        const int ka = zero_index(c, z, mu + 41.0 * kT, K, false), kb = zero_index(c, z, mu - 41.0 * kT, K, true);
        double r = 0.0, eb = 0.0, es = 0.0;
        for (int k = ka; k < kb; ++k) {
            const double E = c + z * xk[k];
            const double t = (E - mu) / kT;
            if (t > 40.0) continue;                    // g < 4.3e-18: no density, energy or entropy
            const double wk = w[(long long)k * Nd];
            if (t < -40.0) {                           // g == 1.0 exactly in FP64, entropy term 0
                r += wk;
                eb += 2.0 * wk * E;
                continue;
            }
            // e = e^{-|t|}: g = 1/(1+e) or e/(1+e), and -(g ln g + (1-g) ln(1-g)) = ln(1+e) + |t| e/(1+e)
            const double e = exp(-fabs(t)), d = 1.0 / (1.0 + e), small = e * d;
            const double g = t > 0.0 ? small : d;
            r += wk * g;
            eb += 2.0 * wk * E * g;
            es -= 2.0 * kT * wk * (log1p(e) + fabs(t) * small);
        }
        for (int k = max(ka, kb); k < K; ++k) {        // the rest below mu - 40 kT
            const double wk = w[(long long)k * Nd];
            r += wk;
            eb += 2.0 * wk * (c + z * xk[k]);
        }
        const double rq = 2.0 / h3 * r;
        rho[q] = rq;
        acc[0] += eb;
        acc[1] += es;
        acc[2] += h3 * rq;
    }
    block_reduce<3>(acc, sh);
    if (threadIdx.x == 0) {
        red[3 * blockIdx.x + 0] = acc[0];
        red[3 * blockIdx.x + 1] = acc[1];
        red[3 * blockIdx.x + 2] = acc[2];
        __threadfence();
        last = atomicAdd(count, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    sum_partials<3>(red, gridDim.x, acc, sh);
    if (threadIdx.x == 0) {
        st[F_EB] = acc[0];
        st[F_ES] = acc[1];
        st[F_NEL] = acc[2];
        *count = 0;
    }
}

int enqueue_density(sq_ctx* ctx, const double* chi, const double* zeta, double mu, double kT, double* rho,
                    int mu_from_state)
{
    const int T = node_threads(ctx->g.Nd, ctx->sm_count);
    density_kernel<<<node_blocks(ctx, T), T, 0, ctx->stream>>>(ctx->d_W, chi, zeta, ctx->g.Nd, ctx->npl + 1, mu, kT, ctx->g.h,
                                                               rho, ctx->d_red, ctx->d_count, ctx->d_fermi, mu_from_state);
    ctx->launches++;
    SQ_CUDA_TRY(cudaGetLastError());
    return SQ_OK;
}

int run_density(sq_ctx* ctx, const double* chi, const double* zeta, double mu, double kT, double* rho,
                double* eb, double* es, double* ne)
{
    int rc = enqueue_density(ctx, chi, zeta, mu, kT, rho, 0);
    if (rc) return rc;
    double st[F_NSTATE];
    SQ_CUDA_TRY(cudaMemcpyAsync(st, ctx->d_fermi, sizeof(st), cudaMemcpyDeviceToHost, ctx->stream));
    SQ_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    if (eb) *eb = st[F_EB];
    if (es) *es = st[F_ES];
    if (ne) *ne = st[F_NEL];
    return SQ_OK;
}

}  // namespace sq
