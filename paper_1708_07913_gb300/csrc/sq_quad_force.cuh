// sq_quad_force.cuh -- the nonlocal atomic forces (Section 3.4, Eq.
// Discrete:NLforce; see sq_force_region.cuh for the formula) on the FP32 quad
// kernels: the recurrence of quad_moments_node run to n_pl, with D += c^j t^j
// folded into the gather (D in per-CTA global scratch in the owners' order).
//
// The contraction with the gradient of D runs in FP64, two lanes per clock and
// SM, so it is laid out for few FP64 instructions: D moves to shared memory in
// the current vector's place (whose zero halos are the Dirichlet boundary), a
// warp takes one (candidate, axis), its lanes one support row each, and along a
// row only G_x and DG_x weigh the gradient; the row's y and z factors follow
// once per row.  25^3 regions on a 16^3 grid, n_pl 48, 4096 nodes: the general form
// took 92 ms, this takes 41.5.
#pragma once
#include "sq_force_region.cuh"
#include "sq_quad.cuh"

namespace sq {

struct QuadForceArgs {
    QuadArgs q;
    double grad[FD_NO + 1];          // gradient weights of Eq. FD:Gradient, d = 1..n_o
    double mu, kT;
    const double* ctab;              // cos(j pi (k + 1/2) / (n_pl + 1)), [j][k]
    const long long* nodes;          // nodes to visit (device, validated on the host), or nullptr: all
    long long nq;                    // their number
    float4* D;                       // per CTA: 4 S 2 32 (owners' order)
    double* fpart;                   // per CTA: 3 MAX_CAND, one node's (candidate, axis) contributions
    double* Fcta;                    // per CTA: 3 n_atoms
};

// Shared memory of the coefficients, as a degree of quad_smem_layout whose
// moment sums take as much: the Fermi function at the Chebyshev zeros and the
// coefficients, n_pl + 1 each.
__host__ __device__ inline int quad_force_npl(int npl) { return 2 * ((2 * npl + 2 + 2) / 3); }

template <int M>
__device__ void quad_force_node(const QuadForceArgs& f, unsigned char* smem, uint32_t taddr, long long node, double* Fc)
{
    using G = QGeo<M>;
    __shared__ float2 red[3][QD_NW];
    __shared__ int red_i[QD_NW + 1];
    __shared__ float s_scale[3];                          // diagonal shift, 1/zeta, 2/zeta
    __shared__ double s_dummy;
    const QuadArgs& a = f.q;
    const NLParams<float>& nl = a.r.nl;
    const int npl = a.r.npl, lb = nl.lb, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    QuadCta<M> k(a, smem, taddr, true, quad_force_npl(npl));
    double *s_fk = k.mom, *s_c = s_fk + npl + 1;
    float4* D = f.D + (size_t)blockIdx.x * (4 * G::S * 2 * 32);
    double* fpart = f.fpart + (size_t)blockIdx.x * 3 * MAX_CAND;
    const QuadNode nd(a.r, node);
    const double chq = a.r.chi[node], zq = a.r.zeta[node];

    quad_clear<M>(k, smem);
    tm_sync();
    const int ncand = quad_setup<M>(a, k, nd.qi, nd.qj, nd.qk, red_i);
    {                                                     // is the node inside some candidate's support?
        bool in = false;
        if (tid < ncand) {                                // at most MAX_CAND = QD_NT candidates
            const int4 cr = k.cand[tid];
            const AtomTab at = nl.atoms[cr.x];
            const int jj = M - cr.z, kk = M - cr.w;
            int xlo, xhi;
            in = jj >= 0 && jj < at.len[1] && kk >= 0 && kk < at.len[2] &&
                 nl_row_interval<float, M>(nl, cr.x, cr.y, jj, kk, xlo, xhi) && xlo <= M && M <= xhi;
        }
        if (!__syncthreads_or(in)) return;
    }
    // c^j = (2/(n_pl+1)) sum_k g(chi + zeta x_k) T_j(x_k), c^0 halved; x_k = T_1(x_k)
    for (int i = tid; i <= npl; i += QD_NT) s_fk[i] = 1.0 / (1.0 + exp((chq + zq * f.ctab[npl + 1 + i] - f.mu) / f.kT));
    if (tid == 0) {
        s_scale[0] = (float)(-3.0 * a.r.g.w[0] - chq);
        s_scale[1] = (float)(1.0 / zq);
        s_scale[2] = (float)(2.0 / zq);
    }
    __syncthreads();
    for (int j = warp; j <= npl; j += QD_NW) {
        double acc = 0.0;
        for (int i = lane; i <= npl; i += 32) acc += s_fk[i] * f.ctab[(size_t)j * (npl + 1) + i];
        acc = warp_sum(acc);
        if (lane == 0) s_c[j] = (j == 0 ? 1.0 : 2.0) / (npl + 1) * acc;
    }
    quad_potential<M>(a, k, nd.vwin, s_scale[0]);
    __syncthreads();
    // t^0 = e_q, t^{-1} = 0, D = c^0 t^0
    for (int i = tid; i < 4 * G::S * 2 * 32; i += QD_NT) D[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k.sub == M / 8 && k.zi == 0) {
        float e[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (k.q == M / 4 && k.p == M / 2) e[(M & 1) * 4 + (M & 3)] = 1.f;
        tm_st8(k.tm + M * 8, e);
        tm_wait_st();
    }
    if (tid == 0) k.t[M * G::PL + G::row(M) + M] = 1.f;
    tm_sync();
    if (tid == 0)
        reinterpret_cast<float*>(D)[((((M / 8) * G::S + M) * 2 + (M & 1)) * 32 + M / 2 + 16 * ((M / 4) & 1)) * 4 + (M & 3)] =
            (float)s_c[0];
    tm_sync();
    uint32_t ca = 0, cb = G::S * 8;
    for (int i = 0; i < npl; ++i) {
        quad_sweep<M, false, true>(a, k, ca, cb, s_scale[i == 0 ? 1 : 2], ncand, red, &s_dummy, D, (float)s_c[i + 1]);
        const uint32_t c = ca;
        ca = cb;
        cb = c;
    }
    // D takes the current vector's place in shared memory
    for (int z = k.zi; z < G::S; z += 4) {
        const float4* dz = D + (size_t)((k.sub * G::S + z) * 2) * 32 + k.lane;
        if (k.act) {
            float* b = k.own + z * G::PL;
            *reinterpret_cast<float4*>(b) = dz[0];
            *reinterpret_cast<float4*>(b + G::OB) = dz[32];
        }
    }
    // the candidates that hold the node, in order (k.span is free now)
    int ni = 0;
    {
        bool in = false;
        if (tid < ncand) {
            const int4 cr = k.cand[tid];
            const AtomTab at = nl.atoms[cr.x];
            const int jj = M - cr.z, kk = M - cr.w;
            int xlo, xhi;
            in = jj >= 0 && jj < at.len[1] && kk >= 0 && kk < at.len[2] &&
                 nl_row_interval<float, M>(nl, cr.x, cr.y, jj, kk, xlo, xhi) && xlo <= M && M <= xhi;
        }
        const int at = block_excl_scan<QD_NW>(in ? 1 : 0, red_i, ni);
        if (in) k.span[at] = tid;
    }
    __syncthreads();
    // one warp per (candidate, axis): -4 sum_comp coef chi'(q) <chi', grad_axis D>
    for (int task = warp; task < 3 * ni; task += QD_NW) {
        const int c = k.span[task / 3], ax = task % 3;
        const int4 cr = k.cand[c];
        const float* Gt = nl.G + (size_t)cr.x * 3 * lb;
        const float* Dt = nl.DG + (size_t)cr.x * 3 * lb;
        const float4* ent = k.ent + (size_t)c * a.recs;
        const int n = k.nent[c];
        double ss = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
        for (int e0 = 0; e0 < n; e0 += 32) {
            const bool on = e0 + lane < n;
            const uint32_t w = on ? __float_as_uint(ent[e0 + lane].x) : 1u << 14;      // beyond the list: an empty row
            const int off = (int)(w & 16383u) * 4, xlo = (w >> 14) & 31, xhi = (w >> 19) & 31;
            const int z = off / G::PL, rem = off - z * G::PL;
            const bool odd = rem >= G::OB;
            const int y = odd ? 2 * ((rem - G::OB) / G::PX) + 1 : 2 * (rem / G::PX);
            const float* row = k.t + off;
            int dp[FD_NO + 1], dm[FD_NO + 1];             // offsets of the neighbours at +d and -d
            float mp[FD_NO + 1], mm[FD_NO + 1];           // 0: beyond the region along z
#pragma unroll
            for (int d = 1; d <= FD_NO; ++d) {
                mp[d] = mm[d] = 1.f;
                if (ax == 0) {
                    dp[d] = d;
                    dm[d] = -d;
                } else if (ax == 1) {
                    dp[d] = odd ? G::row(1 + d) - G::row(1) : G::row(d);
                    dm[d] = odd ? G::row(1 - d) - G::row(1) : G::row(-d);
                } else {
                    const bool up = z + d < G::S, dn = z >= d;
                    dp[d] = up ? d * G::PL : 0;
                    dm[d] = dn ? -d * G::PL : 0;
                    mp[d] = up ? 1.f : 0.f;
                    mm[d] = dn ? 1.f : 0.f;
                }
            }
            double u = 0.0, v = 0.0;
            const int len = __reduce_max_sync(0xffffffffu, xlo <= xhi ? (unsigned)(xhi - xlo + 1) : 0u);
            for (int s = 0; s < len; ++s) {
                const int x = xlo + s;
                if (x <= xhi) {
                    double gd = 0.0;
#pragma unroll
                    for (int d = 1; d <= FD_NO; ++d)
                        gd += f.grad[d] * ((double)(row[x + dp[d]] * mp[d]) - (double)(row[x + dm[d]] * mm[d]));
                    u += (double)Gt[x - cr.y] * gd;
                    v += (double)Dt[x - cr.y] * gd;
                }
            }
            if (on) {
                const double gy = Gt[lb + y - cr.z], dgy = Dt[lb + y - cr.z];
                const double gz = Gt[2 * lb + z - cr.w], dgz = Dt[2 * lb + z - cr.w];
                const double yz = gy * gz;
                ss += u * yz;
                sx += v * yz;
                sy += u * (dgy * gz);
                sz += u * (gy * dgz);
            }
        }
        ss = warp_sum(ss);
        sx = warp_sum(sx);
        sy = warp_sum(sy);
        sz = warp_sum(sz);
        if (lane == 0) {
            const int i0 = M - cr.y, j0 = M - cr.z, k0 = M - cr.w;
            const double g0x = Gt[i0], g0y = Gt[lb + j0], g0z = Gt[2 * lb + k0];
            const double s0 = g0x * g0y * g0z;
            const double x0 = (double)Dt[i0] * g0y * g0z;
            const double y0 = g0x * (double)Dt[lb + j0] * g0z;
            const double z0 = g0x * g0y * (double)Dt[2 * lb + k0];
            fpart[task] = -4.0 * ((double)nl.cs * s0 * ss + (double)nl.cp * (x0 * sx + y0 * sy + z0 * sz));
        }
    }
    __syncthreads();
    if (tid < 3)                                          // one thread per axis, candidates in order
        for (int i = 0; i < ni; ++i) Fc[3 * k.cand[k.span[i]].x + tid] += fpart[3 * i + tid];
    __syncthreads();
}

template <int M>
__global__ void __launch_bounds__(QD_NT, 1) quad_force_kernel(const __grid_constant__ QuadForceArgs f)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_taddr;
    const uint32_t taddr = quad_tmem_alloc(&s_taddr);
    double* Fc = f.Fcta + (size_t)blockIdx.x * 3 * f.q.r.nl.n_atoms;
    for (int i = threadIdx.x; i < 3 * f.q.r.nl.n_atoms; i += QD_NT) Fc[i] = 0.0;
    __syncthreads();
    for (long long iq = blockIdx.x; iq < f.nq; iq += gridDim.x) {
        quad_force_node<M>(f, smem_raw, taddr, f.nodes ? f.nodes[iq] : iq, Fc);
        __syncthreads();
    }
    quad_tmem_free(taddr);
}

}  // namespace sq
