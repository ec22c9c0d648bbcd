// sq_quad.cuh -- FP32 region kernels on quads of points: Lanczos spectral
// bounds and the Chebyshev recurrence with moments (Section 3.2, Eqs. Rec:FD
// and rhoqj), one node per CTA and one CTA of 16 warps per SM.
//
// What bounds a region step is the shared-memory pipe: a point of the
// 37-point stencil read as 24 x/y neighbours of 4 bytes costs 24 of its 32-lane
// wavefronts per 32 points.  Here a thread owns two rows (2p, 2p+1) of a quad
// of four x points.  A plane then costs it 8 LDS.128 for the x windows of both
// rows and 12 for the y neighbours that they share: 10 wavefronts per 32
// points.  The z neighbours, the point itself and the second vector never touch
// shared memory: both recurrence vectors also live in tensor memory (TMEM, 256
// KB per SM, ~740 B/clk measured beside the 128 B/clk of shared memory), in the
// lanes of the thread that owns the points, z along the columns.  Only the
// current vector sits in shared memory, which also makes room for every
// projector table (31^3 keeps two of them in global scratch).
//
// Sums and differences of the stencil run in pairs (add/fma.rn.f32x2: the same
// FP32 rate, half the issue slots) in the order of the general form, so without
// projectors the vectors agree with it bit for bit.
//
// Ownership: warp w reads TMEM lanes 32 (w & 3) .. + 31; lane = p + 16 hf owns
// rows 2p and 2p+1 of quad q = 2 (w & 3) + hf on the planes z = (w >> 2) + 4 j.
// Rows are stored with the even ones first and the odd ones after them, so that
// lanes p, p+1, .. read consecutive stored rows for every neighbour offset; the
// row pitch is an odd multiple of 4 floats, which makes those LDS.128 free of
// bank conflicts.  At least 6 zero columns end every row and 3 zero rows every
// half plane: they are the zero Dirichlet halo (Section 3.1) of both sides.
//
// The projector term is gathered, not scattered: for every (quad, row pair,
// plane) a list of the candidates whose support touches it, built once per
// node, with an 8-bit mask of the points inside.  The inner products are taken
// candidate by candidate, two entries (support rows) per lane.  Every sum has a
// fixed order: results repeat bit for bit.
#pragma once
#include "sq_queue.cuh"
#include "sq_region.cuh"

namespace sq {

constexpr int QD_MMAX = 15;                  // region half-widths 7 .. 15 have a quad kernel
// From these half-widths on a context takes it.  Speed: one node per SM and a
// thread per (quad, row pair) leave lanes and issue slots idle in small regions,
// of which the general kernels keep several per SM; moments, general against quad
// kernel, cycles of one SM per node and step: with projectors 20.3K / 20.7K at
// 13^3, 45.1K / 29.6K at 17^3, 127K / 64K at 29^3; local 7.2K / 9.2K at 13^3,
// 14.6K / 11.8K at 17^3, 37.3K / 18.4K at 29^3.
// Lanczos with projectors besides: in small regions extreme Ritz values that 40
// FP32 steps leave unconverged move with the rounding, and the moments with them
// (largest change over the moments' rms between the two kernels, seven seeded
// systems each: 1e-2 at 17^3, 2e-3 at 19^3, 5e-4 at 21^3, 8e-5 at 23^3, 2e-5 at
// 29^3; 5e-6 at most without projectors).  Those stay on the general kernel, whose
// own run-to-run spread is ten times smaller, so that results there stay what they
// were.  It is no more exact: rms error of zeta against FP64 Lanczos over the rms
// of zeta, seven seeded systems each, general / quad: 1.94e-5 / 1.93e-5 at 15^3,
// 1.02e-5 / 0.98e-5 at 17^3, 8.6e-6 / 8.8e-6 at 19^3, 6.4e-6 / 6.4e-6 at 21^3,
// 3.6e-6 / 3.6e-6 at 23^3; largest error 3.5e-3 / 3.6e-3 at 15^3, 7.8e-5 / 6.9e-5 at
// 23^3.
constexpr int QD_MIN_NL = 7, QD_MIN_LOCAL = 8, QD_MIN_NL_LANCZOS = 11;
constexpr bool quad_has_lanczos(int m) { return m >= QD_MIN_LOCAL || m >= QD_MIN_NL_LANCZOS; }
constexpr int QD_NT = 512, QD_NW = 16;
constexpr int QD_KMAX = 4 * ENTRIES_PER_ROW;  // list length per (quad, row pair, plane pair): four full rows
constexpr int QD_ZERO = 504;                  // 8 TMEM columns of zeros: the planes beyond the region

template <int M>
struct QGeo {
    static constexpr int S = 2 * M + 1, NQ = (S + 3) / 4;
    static constexpr int E = M + 1, OD = M;                       // even and odd rows of a plane
    static constexpr int NP = M + 1;                              // pairs of planes
    static constexpr int PX = ((S + 9) / 8) * 8 + 4;              // >= S + 6, odd multiple of 4
    static constexpr int PAD = ((16 - (E + 3) * PX % 32) + 32) % 32;   // odd rows start half a bank cycle off
    static constexpr int OB = (E + 3) * PX + PAD;                 // first odd row
    static constexpr int PL = OB + (OD + 3) * PX;
    static constexpr int LEAD = 3 * PX + 8, TAIL = PX + 16;
    static constexpr int TF = LEAD + S * PL + TAIL;               // floats of the vector
    static constexpr bool TG = M == 15;                           // y and z tables in global scratch
    __host__ __device__ static constexpr int row(int y) { return (y & 1 ? OB : 0) + (y >> 1) * PX; }
    static_assert(PX >= S + 6 && PX % 8 == 4 && 2 * S * 8 <= QD_ZERO && TF / 4 < (1 << 14), "quad layout");
};

struct QuadArgs {
    RegionArgs<float> r;
    float2 wd2[FD_NO + 1];           // (wd, wd)
    float diag;                      // -3 w_0, the diagonal of the Laplacian term
    char* scratch;                   // per CTA: QuadScratch
    size_t stride;
    const uint32_t* mask;            // [atom][lb planes][lb rows]: columns of a support row, bit i = box column i
    int nxq, nyp, recs;              // per candidate: x quads, row pairs, entry slots
};

// Per-candidate table sizes for boxes of up to lb points per axis.
__host__ __device__ inline int quad_nxq(int lb) { return (lb + 2) / 4 + 1; }
__host__ __device__ inline int quad_nyp(int lb) { return lb / 2 + 1; }
__host__ __device__ inline int quad_recs(int lb) { return (lb * lb + 63) / 64 * 64; }

struct QuadScratch {
    size_t V, list, ent, yt, ab, total;
};
__host__ __device__ inline QuadScratch quad_scratch(int m, int ccap, int lb)
{
    const int S = 2 * m + 1;
    QuadScratch L;
    size_t o = 0;
    L.V = o;     o = align256(o + (size_t)4 * S * 2 * 32 * 16);
    L.list = o;  o = align256(o + (size_t)4 * (m + 1) * QD_KMAX * 32 * 8);
    L.ent = o;   o = align256(o + (size_t)ccap * quad_recs(lb) * 16);
    L.yt = o;    o = align256(o + (m == QD_MMAX ? (size_t)ccap * quad_nyp(lb) * 16 : 0));
    L.ab = o;    o = align256(o + (m == QD_MMAX ? (size_t)(ccap * (lb + 1) + 1) * 16 : 0));
    L.total = ccap > 0 ? o : L.list;     // without projectors only the potential
    return L;
}

// Shared memory after the vector.
struct QuadSmem {
    size_t xq, yt, ab, cand, clen, seg, unit, nent, nvis, span, mom, total;
};
__host__ __device__ inline QuadSmem quad_smem_layout(int m, bool has_nl, int ccap, int lb, int npl)
{
    QuadSmem L;
    size_t o = 0;
    const bool tg = m == QD_MMAX;
    L.xq = L.yt = L.ab = L.cand = L.clen = L.seg = L.unit = L.nent = L.nvis = L.span = 0;
    if (has_nl) {
        L.xq = o;    o = align16(o + (size_t)ccap * quad_nxq(lb) * 32);
        L.yt = o;    o = align16(o + (tg ? 0 : (size_t)ccap * quad_nyp(lb) * 16));
        L.ab = o;    o = align16(o + (tg ? 0 : (size_t)(ccap * (lb + 1) + 1) * 16));
        L.cand = o;  o = align16(o + (size_t)ccap * 16);
        L.seg = o;   o = align16(o + (size_t)(ccap + QD_NW) * 16);
        L.clen = o;  o = align16(o + (size_t)ccap * 4);
        L.unit = o;  o = align16(o + (size_t)(ccap + 1) * 4);
        L.nent = o;  o = align16(o + (size_t)ccap * 4);
        L.nvis = o;  o = align16(o + (size_t)4 * (m + 1) * 4);
        L.span = L.clen;                     // the box lengths are not needed after the set-up
    }
    L.mom = o;
    if (npl > 0) o = align16(o + (size_t)3 * (npl / 2 + 2) * sizeof(double));
    L.total = o;
    return L;
}
template <int M>
__host__ __device__ inline size_t quad_smem_bytes(bool has_nl, int ccap, int lb, int npl)
{
    return (size_t)QGeo<M>::TF * 4 + quad_smem_layout(M, has_nl, ccap, lb, npl).total;
}

// ---- pairs of floats -------------------------------------------------------
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float lo2(f2 a)
{
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
    return x;
}
__device__ __forceinline__ float hi2(f2 a)
{
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
    return y;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// ---- tensor memory: 8 columns of this thread's lane -------------------------
__device__ __forceinline__ void tm_ld8(uint32_t a, float (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "r"(a));
}
__device__ __forceinline__ void tm_st8(uint32_t a, const float (&v)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};"
                 ::"f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "r"(a));
}
// The loads issued so far have arrived: their registers pass through the wait
// (tm_ready for the second and later ones), so no use moves above it.
__device__ __forceinline__ void tm_wait_ld(float (&v)[8])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]));
}
__device__ __forceinline__ void tm_ready(float (&v)[8])
{
    asm volatile("" : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]));
}
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// CTA barrier that also orders the tensor-memory accesses of the warps
__device__ __forceinline__ void tm_sync()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Sum of one float per thread over the CTA: compensated FP32 trees (value and
// running error) within the warps and then over their 16 results, so that FP64,
// two lanes per clock on this part, is left with one addition per sum.  Every
// warp calls quad_warp_sums before the barrier; quad_cta_sums after it, by the
// whole of one warp, leaves the totals in its lane 0.
template <int N>
__device__ __forceinline__ void quad_warp_sums(const float (&v)[N], float2 (*red)[QD_NW])
{
    float s[N], c[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        s[i] = v[i];
        c[i] = 0.f;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        float t[N], tc[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {                     // the trees side by side
            t[i] = __shfl_xor_sync(0xffffffffu, s[i], o);
            tc[i] = __shfl_xor_sync(0xffffffffu, c[i], o);
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            float e;
            two_sum(s[i], t[i], s[i], e);
            c[i] = c[i] + (tc[i] + e);
        }
    }
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int i = 0; i < N; ++i) red[i][threadIdx.x >> 5] = make_float2(s[i], c[i]);
}
template <int N>
__device__ __forceinline__ void quad_cta_sums(const float2 (*red)[QD_NW], double (&out)[N])
{
    float s[N], c[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const float2 r = red[i][threadIdx.x & 15];
        s[i] = r.x;
        c[i] = r.y;
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
        float t[N], tc[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            t[i] = __shfl_xor_sync(0xffffffffu, s[i], o);
            tc[i] = __shfl_xor_sync(0xffffffffu, c[i], o);
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            float e;
            two_sum(s[i], t[i], s[i], e);
            c[i] = c[i] + (tc[i] + e);
        }
    }
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int i = 0; i < N; ++i) out[i] = (double)s[i] + (double)c[i];
}

// Streamed global loads that leave the L1 to the tables.
__device__ __forceinline__ float4 ldg_stream4(const float4* p)
{
    float4 v;
    asm volatile("ld.global.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ldg_stream2(const uint2* p)
{
    uint2 v;
    asm volatile("ld.global.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 lds4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
// A list entry: addresses of the x profiles, of the row pair's y factors and of
// the first plane's coefficients (multiples of 16 below 2^18: bits 4-17 of x,
// 18-31 of x, 2-15 of y; shared memory, or offsets into global scratch where
// those tables are), and the points inside the support (bits 16-31 of y: 4 per
// row; row 2p and 2p+1 of the first plane, then of the second).
__device__ __forceinline__ uint2 quad_entry(uint32_t x, uint32_t y, uint32_t ab, uint32_t nib)
{
    return make_uint2(x | (y << 14), (ab >> 2) | (nib << 16));
}

// Arguments of the quad kernels with the region arguments a.
inline QuadArgs quad_args(const sq_ctx* c, const RegionArgs<float>& a)
{
    QuadArgs q;
    memset(&q, 0, sizeof(q));
    q.r = a;
    for (int d = 0; d <= FD_NO; ++d) q.wd2[d] = make_float2(a.wd[d], a.wd[d]);
    q.diag = (float)(-3.0 * c->g.w[0]);
    q.scratch = (char*)c->d_qscratch;
    q.stride = c->q_stride;
    q.mask = c->d_qmask;
    q.nxq = quad_nxq(c->lb);
    q.nyp = quad_nyp(c->lb);
    q.recs = quad_recs(c->lb);
    return q;
}

// Where one CTA keeps things, and what one thread owns.
template <int M>
struct QuadCta {
    using G = QGeo<M>;
    float* t;                        // the current vector (LEAD floats in: region row 0, plane 0)
    float4 *xq, *yt, *ab, *seg, *V;
    int4* cand;
    int *clen, *unit, *nent, *nvis, *span;
    uint2* list;
    float4* ent;
    double* mom;
    uint32_t tm;                     // tensor memory, lanes of this warp
    int sub, zi, lane, p, q;
    bool act;                        // owns points
    float* own;                      // t of (row 2p, quad q, plane 0); idle lanes: of a neighbour that does

    __device__ QuadCta(const QuadArgs& a, unsigned char* smem, uint32_t taddr, bool has_nl, int npl)
    {
        const int tid = threadIdx.x, w = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform
        lane = tid & 31;
        sub = w & 3;
        zi = w >> 2;
        p = lane & 15;
        q = 2 * sub + (lane >> 4);
        act = p < G::E && q < G::NQ;
        tm = taddr + ((uint32_t)(sub * 32) << 16);
        t = reinterpret_cast<float*>(smem) + G::LEAD;
        const int pc = p < G::E ? p : G::E - 1, qc = q < G::NQ ? q : (2 * sub < G::NQ ? 2 * sub : 0);
        own = t + pc * G::PX + 4 * qc;
        unsigned char* b = smem + (size_t)G::TF * 4;
        const QuadSmem L = quad_smem_layout(M, has_nl, a.r.nl.ccap, a.r.nl.lb, npl);
        char* g = a.scratch + (size_t)blockIdx.x * a.stride;
        const QuadScratch Q = quad_scratch(M, has_nl ? a.r.nl.ccap : 0, has_nl ? a.r.nl.lb : 0);
        xq = reinterpret_cast<float4*>(b + L.xq);
        yt = G::TG ? reinterpret_cast<float4*>(g + Q.yt) : reinterpret_cast<float4*>(b + L.yt);
        ab = G::TG ? reinterpret_cast<float4*>(g + Q.ab) : reinterpret_cast<float4*>(b + L.ab);
        seg = reinterpret_cast<float4*>(b + L.seg);
        cand = reinterpret_cast<int4*>(b + L.cand);
        clen = reinterpret_cast<int*>(b + L.clen);
        unit = reinterpret_cast<int*>(b + L.unit);
        nent = reinterpret_cast<int*>(b + L.nent);
        nvis = reinterpret_cast<int*>(b + L.nvis);
        span = reinterpret_cast<int*>(b + L.span);
        mom = reinterpret_cast<double*>(b + L.mom);
        V = reinterpret_cast<float4*>(g + Q.V);
        list = reinterpret_cast<uint2*>(g + Q.list);
        ent = reinterpret_cast<float4*>(g + Q.ent);
    }
};

// The first entries of all three tables, no points.
template <int M>
__device__ __forceinline__ uint2 quad_none(const QuadCta<M>& k)
{
    return quad_entry((uint32_t)__cvta_generic_to_shared(k.xq), QGeo<M>::TG ? 0u : (uint32_t)__cvta_generic_to_shared(k.yt),
                      QGeo<M>::TG ? 0u : (uint32_t)__cvta_generic_to_shared(k.ab), 0u);
}

// The potential window of the node plus the diagonal shift, in owner order.
template <int M>
__device__ void quad_potential(const QuadArgs& a, const QuadCta<M>& k, const float* vwin, float dshift)
{
    using G = QGeo<M>;
    const size_t plane = (size_t)a.r.g.P1 * a.r.g.P2;
    for (int z = k.zi; z < G::S; z += 4)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int y = 2 * k.p + r;
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            if (k.act && y < G::S) {
                const float* src = vwin + (size_t)z * plane + (size_t)y * a.r.g.P1 + 4 * k.q;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (4 * k.q + i < G::S) v[i] = src[i] + dshift;
            }
            k.V[(size_t)((k.sub * G::S + z) * 2 + r) * 32 + k.lane] = make_float4(v[0], v[1], v[2], v[3]);
        }
}

// Columns xlo..xhi of a support row as a bit mask (region columns).
__device__ __forceinline__ uint32_t col_mask(int xlo, int xhi) { return (0xffffffffu >> (31 - xhi)) & (0xffffffffu << xlo); }

// Projector bookkeeping for one node: candidates (atom images of the node's
// tile whose box meets the region, in tile-list order), their x and y tables
// aligned to the region's quads and row pairs, the entries (support rows) by
// candidate for the inner products, and the lists by (quad, row pair, plane)
// for the gather.  No region row has more than ENTRIES_PER_ROW entries (contexts
// with such a row keep the general kernels, which refuse them).  Returns the
// candidate count.
template <int M>
__device__ int quad_setup(const QuadArgs& a, const QuadCta<M>& k, int qi, int qj, int qk, int* red_i)
{
    using G = QGeo<M>;
    const NLParams<float>& nl = a.r.nl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int lb = nl.lb;
    const int tile = (qi / TILE) + nl.ntile[0] * ((qj / TILE) + nl.ntile[1] * (qk / TILE));
    const int beg = nl.tile_start[tile], end = nl.tile_start[tile + 1];
    int ncand = 0;
    for (int c0 = beg; c0 < end; c0 += QD_NT) {
        const int c = c0 + tid;
        int keep = 0, ln = 0;
        int4 rec = make_int4(0, 0, 0, 0);
        if (c < end) {
            const int4 tc = nl.tile_cand[c];
            const AtomTab at = nl.atoms[tc.x];
            const int bx = tc.y - (qi - M), by = tc.z - (qj - M), bz = tc.w - (qk - M);
            keep = (bx < G::S && bx + at.len[0] > 0 && by < G::S && by + at.len[1] > 0 && bz < G::S &&
                    bz + at.len[2] > 0);
            rec = make_int4(tc.x, bx, by, bz);
            ln = at.len[0] | (at.len[1] << 8) | (at.len[2] << 16);
        }
        int tot;
        const int pos = block_excl_scan<QD_NW>(keep, red_i, tot);
        if (keep) {
            if (ncand + pos < nl.ccap) {
                k.cand[ncand + pos] = rec;
                k.clen[ncand + pos] = ln;
            } else {
                atomicOr(a.r.err, ERR_CAPACITY);
            }
        }
        ncand += tot;
    }
    if (ncand > nl.ccap) ncand = nl.ccap;
    __syncthreads();
    // x tables: quads q0 + j of the region, q0 = floor(bx / 4), zero beyond the box
    for (int i = tid; i < ncand * a.nxq; i += QD_NT) {
        const int c = i / a.nxq, j = i % a.nxq;
        const int4 cr = k.cand[c];
        const int lx = k.clen[c] & 255;
        const float* Gt = nl.G + (size_t)cr.x * 3 * lb;
        const float* Dt = nl.DG + (size_t)cr.x * 3 * lb;
        float g[4], d[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int col = 4 * ((cr.y >> 2) + j) + e - cr.y;
            const bool in = col >= 0 && col < lx;
            g[e] = in ? Gt[col] : 0.f;
            d[e] = in ? Dt[col] : 0.f;
        }
        k.xq[2 * i] = make_float4(g[0], g[1], g[2], g[3]);
        k.xq[2 * i + 1] = make_float4(d[0], d[1], d[2], d[3]);
    }
    // y tables: (G_y, DG_y) of the row pairs p0 + j, p0 = floor(by / 2)
    for (int i = tid; i < ncand * a.nyp; i += QD_NT) {
        const int c = i / a.nyp, j = i % a.nyp;
        const int4 cr = k.cand[c];
        const int ly = (k.clen[c] >> 8) & 255;
        const float* Gt = nl.G + ((size_t)cr.x * 3 + 1) * lb;
        const float* Dt = nl.DG + ((size_t)cr.x * 3 + 1) * lb;
        const int j0 = 2 * ((cr.z >> 1) + j) - cr.z, j1 = j0 + 1;
        const bool in0 = j0 >= 0 && j0 < ly, in1 = j1 >= 0 && j1 < ly;
        k.yt[i] = make_float4(in0 ? Gt[j0] : 0.f, in0 ? Dt[j0] : 0.f, in1 ? Gt[j1] : 0.f, in1 ? Dt[j1] : 0.f);
    }
    // lists: every thread its own (quad, row pair), a warp every fourth pair of planes; per pair the candidates
    // that meet it and the warp's quads, in order, six candidates' support rows in flight
    {
        const uint2 none = quad_none<M>(k);
        const uint32_t xb = none.x & 0x3fff0u, yb = (none.x >> 14) & 0x3fff0u, bb = (none.y << 2) & 0x3fff0u;
        const int y0 = 2 * k.p, xw = 8 * k.sub;
        const uint32_t cols = 4 * k.q + 4 <= G::S ? 15u : 15u >> (4 * k.q + 4 - G::S);      // the quad's region columns
        for (int zp = k.zi; zp < G::NP; zp += 4) {
            const int z = 2 * zp;
            uint2* lp = k.list + (size_t)(k.sub * G::NP + zp) * QD_KMAX * 32 + k.lane;
            int n = 0;
            for (int cb = 0; cb < ncand; cb += 32) {
                const int ct = cb + lane;
                bool hit = false;
                if (ct < ncand) {
                    const int4 cr = k.cand[ct];
                    const int ln = k.clen[ct];
                    hit = cr.w <= z + 1 && cr.w + (ln >> 16) > z && cr.y < xw + 8 && cr.y + (ln & 255) > xw;
                }
                unsigned set = __ballot_sync(0xffffffffu, hit);
                while (set) {                             // warp-uniform
                    int cc[6];
                    uint32_t m[6][4];
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        cc[i] = set ? cb + __ffs(set) - 1 : -1;
                        set &= set - 1;
                        m[i][0] = m[i][1] = m[i][2] = m[i][3] = 0;
                        if (cc[i] < 0) continue;
                        const int4 cr = k.cand[cc[i]];
                        const int ln = k.clen[cc[i]];
                        const int jj = y0 - cr.z, kk = z - cr.w, ly = (ln >> 8) & 255, lz = ln >> 16;
                        const uint32_t* src = a.mask + ((ptrdiff_t)cr.x * lb + kk) * lb + jj;
                        const bool r0 = k.act && jj >= 0 && jj < ly, r1 = k.p < G::OD && k.act && jj >= -1 && jj + 1 < ly;
                        const bool p0 = kk >= 0, p1 = kk + 1 < lz && z + 1 < G::S;
                        if (r0 && p0) m[i][0] = src[0];
                        if (r1 && p0) m[i][1] = src[1];
                        if (r0 && p1) m[i][2] = src[lb];
                        if (r1 && p1) m[i][3] = src[lb + 1];
                    }
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        if (cc[i] < 0) break;
                        const int4 cr = k.cand[cc[i]];
                        const int sh = 4 * k.q - cr.y;        // region column 4q is box column sh
                        uint32_t nib = 0;
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            nib |= ((sh >= 0 ? m[i][e] >> min(sh, 31) : m[i][e] << min(-sh, 31)) & cols) << (4 * e);
                        if (sh >= 32 || sh <= -32) nib = 0;
                        if (nib) {
                            if (n < QD_KMAX)
                                lp[n * 32] = quad_entry(xb + (uint32_t)(cc[i] * a.nxq + k.q - (cr.y >> 2)) * 32u,
                                                        yb + (uint32_t)(cc[i] * a.nyp + k.p - (cr.z >> 1)) * 16u,
                                                        bb + (uint32_t)(cc[i] * (lb + 1) + 1 + z - cr.w) * 16u, nib);
                            ++n;
                        }
                    }
                    __syncwarp();
                }
            }
            // the longest list, made even; shorter ones and idle lanes end in entries without points
            int most = min(__reduce_max_sync(0xffffffffu, (unsigned)n), (unsigned)QD_KMAX);
            most += most & 1;
            if (lane == 0) k.nvis[k.sub * G::NP + zp] = most;
            for (; n < most; ++n) lp[n * 32] = none;
        }
    }
    // entries: warp per candidate, its box rows clipped to the region, compacted with a ballot
    for (int c = warp; c < ncand; c += QD_NW) {
        const int4 cr = k.cand[c];
        const int ln = k.clen[c];
        const float* Gt = nl.G + (size_t)cr.x * 3 * lb;
        const float* Dt = nl.DG + (size_t)cr.x * 3 * lb;
        const int j0 = max(0, -cr.z), j1 = min((ln >> 8) & 255, G::S - cr.z);
        const int k0 = max(0, -cr.w), k1 = min(ln >> 16, G::S - cr.w);
        const int nj = j1 - j0, nrows = (nj > 0 && k1 > k0) ? nj * (k1 - k0) : 0;
        const int inv = nj > 0 ? (65535 + nj) / nj : 0;
        float4* out = k.ent + (size_t)c * a.recs;
        int cnt = 0;
        for (int r0 = 0; r0 < nrows; r0 += 96) {           // the loads of three rows per lane are in flight together
            bool ok[3];
            int xlo[3], xhi[3], off[3];
            float gy[3], dgy[3], gz[3], dgz[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int rr = r0 + 32 * i + lane;
                ok[i] = false;
                if (rr < nrows) {
                    const int dk = (rr * inv) >> 16;          // rr / nj, exact for rr < 1024 and nj <= 32
                    const int jj = j0 + rr - dk * nj, kk = k0 + dk;
                    const uint32_t mk = a.mask[((size_t)cr.x * lb + kk) * lb + jj];
                    xlo[i] = max(cr.y + __ffs(mk) - 1, 0);
                    xhi[i] = min(cr.y + 31 - __clz(mk), G::S - 1);
                    ok[i] = mk != 0 && xlo[i] <= xhi[i];
                    off[i] = (cr.w + kk) * G::PL + G::row(cr.z + jj);
                    gy[i] = Gt[lb + jj];
                    dgy[i] = Dt[lb + jj];
                    gz[i] = Gt[2 * lb + kk];
                    dgz[i] = Dt[2 * lb + kk];
                }
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const unsigned bal = __ballot_sync(0xffffffffu, ok[i]);
                if (ok[i])
                    out[cnt + __popc(bal & ((1u << lane) - 1u))] = make_float4(
                        __uint_as_float((uint32_t)(off[i] >> 2) | ((uint32_t)xlo[i] << 14) | ((uint32_t)xhi[i] << 19)),
                        gy[i] * gz[i], dgy[i] * gz[i], gy[i] * dgz[i]);
                cnt += __popc(bal);
            }
        }
        if (lane == 0) k.nent[c] = cnt;
    }
    __syncthreads();
    // units of 64 entries: offsets by candidate
    {
        int run = 0;
        for (int c0 = 0; c0 < ncand; c0 += QD_NT) {
            const int c = c0 + tid;
            int tot;
            const int off = block_excl_scan<QD_NW>(c < ncand ? (k.nent[c] + 63) >> 6 : 0, red_i, tot);
            if (c < ncand) k.unit[c] = run + off;
            run += tot;
        }
        if (tid == 0) k.unit[ncand] = run;
        __syncthreads();
        const int Q = max(1, (run + QD_NW - 1) / QD_NW);  // units of one warp
        for (int c = tid; c < ncand; c += QD_NT) {
            const int f0 = k.unit[c], f1 = k.unit[c + 1];
            k.span[c] = f1 > f0 ? f0 / Q | (((f1 - 1) / Q + 1) << 8) : 0;
        }
    }
    __syncthreads();
    return ncand;
}

// One quad of an entry's row against the candidate's x profiles.
__device__ __forceinline__ void quad_dot(uint32_t nib, const float4& t, const float4& g, const float4& d, float& u, float& v)
{
    if (nib & 1u) { u += g.x * t.x; v += d.x * t.x; }
    if (nib & 2u) { u += g.y * t.y; v += d.y * t.y; }
    if (nib & 4u) { u += g.z * t.z; v += d.z * t.z; }
    if (nib & 8u) { u += g.w * t.w; v += d.w * t.w; }
}

// Projector inner products of the current vector (trapezoidal rule, Eq.
// IntApprox, without the h^3 which sits in cs/cp): S, X, Y, Z of every
// candidate.  A unit is 64 entries of one candidate, two per lane, which share
// the candidate's x profiles (loads with one address per warp); every warp
// takes an equal run of units and leaves its partial sums of candidate c in
// seg[c + warp], distinct for every (candidate, warp) pair that occurs.
template <int M>
__device__ void quad_dots(const QuadArgs& a, const QuadCta<M>& k, int ncand)
{
    using G = QGeo<M>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int U = k.unit[ncand], Q = (U + QD_NW - 1) / QD_NW;
    const int u0 = warp * Q, u1 = min(U, u0 + Q);
    if (u0 >= u1) return;
    int c = 0, hi = ncand - 1;                            // last candidate with unit[c] <= u0
    while (c < hi) {
        const int mid = (c + hi + 1) >> 1;
        if (k.unit[mid] <= u0) c = mid;
        else hi = mid - 1;
    }
    // records of the next two units are in flight while one is summed; cf, first and end follow the fetches
    int cf = c, first = k.unit[c], end = k.unit[c + 1], nf = k.nent[c];
    const float4 none = make_float4(__uint_as_float(1u << 14), 0.f, 0.f, 0.f);    // an empty interval
    auto fetch = [&](int u, float4& r0, float4& r1, int& cc, int& left) {
        r0 = r1 = none;
        cc = cf;
        left = 0;
        if (u >= u1) return;
        while (u >= end) {
            ++cf;
            first = end;
            end = k.unit[cf + 1];
            nf = k.nent[cf];
        }
        cc = cf;
        left = nf - (u - first) * 64;
        const float4* src = k.ent + (size_t)cf * a.recs + (u - first) * 64 + lane;
        if (lane < left) r0 = ldg_stream4(src);
        if (lane + 32 < left) r1 = ldg_stream4(src + 32);
    };
    float4 a0, a1, b0, b1, c0, c1;
    int left, cb, lb2, cn, lc;
    fetch(u0, a0, a1, c, left);
    fetch(u0 + 1, b0, b1, cb, lb2);
    float aS = 0.f, aX = 0.f, aY = 0.f, aZ = 0.f;
    for (int u = u0; u < u1; ++u) {
        fetch(u + 2, c0, c1, cn, lc);
        const uint32_t w0 = __float_as_uint(a0.x), w1 = __float_as_uint(a1.x);
        const int h0 = (w0 >> 19) & 31, l0 = (w0 >> 14) & 31, h1 = (w1 >> 19) & 31, l1 = (w1 >> 14) & 31;
        const uint32_t m0 = l0 <= h0 ? col_mask(l0, h0) : 0u, m1 = l1 <= h1 ? col_mask(l1, h1) : 0u;
        const uint32_t all = __reduce_or_sync(0xffffffffu, m0 | m1);
        const bool two = left > 32;
        const int qa = (__ffs(all) - 1) >> 2, qb = (31 - __clz(all)) >> 2;
        const float4* xq = k.xq + 2 * (c * a.nxq - (k.cand[c].y >> 2));
        const float4* t0 = reinterpret_cast<const float4*>(k.t) + (w0 & 16383u);
        const float4* t1 = reinterpret_cast<const float4*>(k.t) + (w1 & 16383u);
        float s0 = 0.f, d0 = 0.f, s1 = 0.f, d1 = 0.f;
#pragma unroll
        for (int q = 0; q < G::NQ; ++q)                   // region quads: the bit tests are immediates
            if (q >= qa && q <= qb) {                     // warp-uniform
                const float4 g = xq[2 * q], d = xq[2 * q + 1], t = t0[q];
                if (two) {
                    const float4 t2 = t1[q];
                    quad_dot(m0 >> (4 * q), t, g, d, s0, d0);
                    quad_dot(m1 >> (4 * q), t2, g, d, s1, d1);
                } else {
                    quad_dot(m0 >> (4 * q), t, g, d, s0, d0);
                }
            }
        aS += a0.y * s0 + a1.y * s1;
        aX += a0.y * d0 + a1.y * d1;
        aY += a0.z * s0 + a1.z * s1;
        aZ += a0.w * s0 + a1.w * s1;
        if (u + 1 >= u1 || cb != c) {                     // warp-uniform: candidate done in this warp
            // four sums over the warp: two exchanges leave one of them per lane pair bit, three more finish it
            const bool h = lane & 1, h2 = lane & 2;
            const float r0 = (h ? aX : aS) + __shfl_xor_sync(0xffffffffu, h ? aS : aX, 1);
            const float r1 = (h ? aZ : aY) + __shfl_xor_sync(0xffffffffu, h ? aY : aZ, 1);
            float r = (h2 ? r1 : r0) + __shfl_xor_sync(0xffffffffu, h2 ? r0 : r1, 2);
            r += __shfl_xor_sync(0xffffffffu, r, 4);
            r += __shfl_xor_sync(0xffffffffu, r, 8);
            r += __shfl_xor_sync(0xffffffffu, r, 16);
            if (lane < 4) reinterpret_cast<float*>(k.seg + c + warp)[lane] = r;
            aS = aX = aY = aZ = 0.f;
        }
        a0 = b0;
        a1 = b1;
        c = cb;
        left = lb2;
        b0 = c0;
        b1 = c1;
        cb = cn;
        lb2 = lc;
    }
}

// The coefficients of candidate c on plane kk of its box,
//   b0 = G_y alpha + DG_y beta,  b1 = G_y gamma  (a point gets G_x b0 + DG_x b1),
//   alpha = coef (cs G_z S + cp DG_z Z),  beta = coef cp G_z Y,  gamma = coef cp G_z X,
// with the candidate's inner products summed in warp order.  Holds the barrier
// between the inner products and their use.
template <int M>
__device__ void quad_coefs(const QuadArgs& a, const QuadCta<M>& k, int ncand, float coef)
{
    const NLParams<float>& nl = a.r.nl;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lb = nl.lb;
    const float cs = nl.cs * coef, cp = nl.cp * coef;
    // the z profiles of the warp's candidates, eight at a time in flight; the first ones cross the barrier
    // that the inner products need
    for (int c0 = warp; c0 == warp || c0 < ncand; c0 += 8 * QD_NW) {
        float gz[8], dz[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int c = c0 + i * QD_NW;
            gz[i] = dz[i] = 0.f;
            if (c < ncand && lane < lb) {
                const size_t at = ((size_t)k.cand[c].x * 3 + 2) * lb + lane;
                gz[i] = nl.G[at];
                dz[i] = nl.DG[at];
            }
        }
        if (c0 == warp) __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int c = c0 + i * QD_NW;
            if (c >= ncand) break;
            float4 P = make_float4(0.f, 0.f, 0.f, 0.f);
            const int span = k.span[c];                   // the warps that reduced part of it
            for (int w = span & 255; w < span >> 8; ++w) {
                const float4 s = k.seg[c + w];
                P.x += s.x;
                P.y += s.y;
                P.z += s.z;
                P.w += s.w;
            }
            if (lane < lb)
                k.ab[c * (lb + 1) + 1 + lane] =
                    make_float4(cs * gz[i] * P.x + cp * dz[i] * P.w, cp * gz[i] * P.z, cp * gz[i] * P.y, 0.f);
        }
    }
}

// The first QD_AHEAD entries of a list of n (n even; entries beyond it stay what they were).
constexpr int QD_AHEAD = 8;
__device__ __forceinline__ void quad_ahead(const uint2* lp, int n, uint2 (&m)[QD_AHEAD])
{
#pragma unroll
    for (int i = 0; i < QD_AHEAD; i += 2)
        if (i < n) {                                      // warp-uniform
            m[i] = ldg_stream2(lp + i * 32);
            m[i + 1] = ldg_stream2(lp + (i + 1) * 32);
        }
}

// One entry's contribution to the 16 points of a thread (two rows on two planes).
struct QuadTab {
    float4 g, d, y, a0, a1;
};
template <int M>
__device__ __forceinline__ QuadTab quad_tables(const QuadCta<M>& k, const uint2& m)
{
    const uint32_t xa = m.x & 0x3fff0u, ya = (m.x >> 14) & 0x3fff0u, aa = (m.y << 2) & 0x3fff0u;
    QuadTab t;
    if constexpr (QGeo<M>::TG) {
        t.y = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(k.yt) + ya);
        t.a0 = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(k.ab) + aa);
        t.a1 = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(k.ab) + aa + 16);
    } else {
        t.y = lds4(ya);
        t.a0 = lds4(aa);
        t.a1 = lds4(aa + 16);
    }
    t.g = lds4(xa);
    t.d = lds4(xa + 16);
    return t;
}
__device__ __forceinline__ void quad_row(uint32_t w, int bit, const float4& g, const float4& d, float gy, float dy,
                                         const float4& ab, float* nl)
{
    const float b0 = gy * ab.x + dy * ab.y, b1 = gy * ab.z;
    if (w & (1u << bit)) { nl[0] += g.x * b0; nl[0] += d.x * b1; }
    if (w & (2u << bit)) { nl[1] += g.y * b0; nl[1] += d.y * b1; }
    if (w & (4u << bit)) { nl[2] += g.z * b0; nl[2] += d.z * b1; }
    if (w & (8u << bit)) { nl[3] += g.w * b0; nl[3] += d.w * b1; }
}
__device__ __forceinline__ void quad_visit(uint32_t w, const QuadTab& t, float (&nl)[16])
{
    quad_row(w, 16, t.g, t.d, t.y.x, t.y.y, t.a0, nl);
    quad_row(w, 20, t.g, t.d, t.y.z, t.y.w, t.a0, nl + 4);
    quad_row(w, 24, t.g, t.d, t.y.x, t.y.y, t.a1, nl + 8);
    quad_row(w, 28, t.g, t.d, t.y.z, t.y.w, t.a1, nl + 12);
}

// The thread's points inside the region, one bit each (row 2p first).
template <int M>
__device__ __forceinline__ uint32_t quad_inside(const QuadCta<M>& k)
{
    using G = QGeo<M>;
    uint32_t in = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) in |= (k.act && 4 * k.q + (i & 3) < G::S && (i < 4 || k.p < G::OD)) ? 1u << i : 0u;
    return in;
}

// Sums of a sweep, two points at a time: out.out, out.t and (Lanczos) t.t.
struct QuadSums {
    f2 aa = 0, ab = 0, ac = 0;
    template <bool TT>
    __device__ __forceinline__ void add(f2 o, f2 t)
    {
        aa = fma2(o, o, aa);
        ab = fma2(o, t, ab);
        if (TT) ac = fma2(t, t, ac);
    }
};

// The local part of one sweep of H over the region: on plane z and both rows of
// the thread
//   out = s [ (V - shift) t - 1/2 sum_d w_d (6 neighbours at d) ] - sec,
// t in columns ca of tensor memory and in shared memory, sec in columns cb,
// which receive out.  FIN: there is no projector term to come: out is cut to
// the region, summed, and its centre value kept.
template <int M, bool TT, bool FIN>
__device__ void quad_stencil(const QuadArgs& a, const QuadCta<M>& k, uint32_t ca, uint32_t cb, float s, QuadSums& sum,
                             double* centre)
{
    using G = QGeo<M>;
    const f2 s2 = pack2(s, s);
    const uint32_t in = FIN ? quad_inside<M>(k) : 0u;
    for (int z = k.zi; z < G::S; z += 4) {
        const float* b = k.own + z * G::PL;
        auto plane = [&](int zz) { return (unsigned)zz < (unsigned)G::S ? k.tm + ca + zz * 8 : k.tm + QD_ZERO; };
        float tc[8], zp[8], zm[8], sc[8];
        tm_ld8(k.tm + ca + z * 8, tc);
        tm_ld8(plane(z + 1), zp);
        tm_ld8(plane(z - 1), zm);
        // x windows: pairs (x-8,x-7) .. (x+10,x+11) of both rows, the own quad at pairs 4 and 5
        f2 X[2][10];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const ulonglong2* w = reinterpret_cast<const ulonglong2*>(b + r * G::OB);
            ulonglong2 u;
            u = w[-2]; X[r][0] = u.x; X[r][1] = u.y;
            u = w[-1]; X[r][2] = u.x; X[r][3] = u.y;
            u = w[1];  X[r][6] = u.x; X[r][7] = u.y;
            u = w[2];  X[r][8] = u.x; X[r][9] = u.y;
        }
        f2 lap[2][2] = {{0ull, 0ull}, {0ull, 0ull}};
        const float4* vp = k.V + (size_t)((k.sub * G::S + z) * 2) * 32 + k.lane;
        float4 v0, v1;
        f2 up[2], dn[2];                                  // rows r0 + d and r1 - d of the previous d
        tm_wait_ld(tc);
        tm_ready(zp);
        tm_ready(zm);
        f2 own[2][2];
        own[0][0] = pack2(tc[0], tc[1]);
        own[0][1] = pack2(tc[2], tc[3]);
        own[1][0] = pack2(tc[4], tc[5]);
        own[1][1] = pack2(tc[6], tc[7]);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int j = 0; j < 2; ++j) X[r][4 + j] = own[r][j];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            up[j] = own[1][j];
            dn[j] = own[0][j];
        }
#pragma unroll
        for (int d = 1; d <= FD_NO; ++d) {
            f2 zs[2][2];
#pragma unroll
            for (int i = 0; i < 4; ++i) zs[i >> 1][i & 1] = add2(pack2(zp[2 * i], zp[2 * i + 1]), pack2(zm[2 * i], zm[2 * i + 1]));
            if (d < FD_NO) {                              // the next planes arrive while this d is summed
                tm_ld8(plane(z + d + 1), zp);
                tm_ld8(plane(z - d - 1), zm);
            } else {
                tm_ld8(k.tm + cb + z * 8, sc);
            }
            const ulonglong2 yl = *reinterpret_cast<const ulonglong2*>(b + G::row(-d));       // row r0 - d
            const ulonglong2 yh = *reinterpret_cast<const ulonglong2*>(b + G::row(d + 1));    // row r1 + d
            const f2 lo[2] = {yl.x, yl.y}, hi[2] = {yh.x, yh.y};
            const f2 wd = *reinterpret_cast<const f2*>(&a.wd2[d]);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    f2 xs;
                    if (d % 2 == 0) {
                        xs = add2(X[r][4 + j + d / 2], X[r][4 + j - d / 2]);
                    } else {
                        xs = pack2(hi2(X[r][4 + j + (d - 1) / 2]) + hi2(X[r][4 + j - (d + 1) / 2]),
                                   lo2(X[r][4 + j + (d + 1) / 2]) + lo2(X[r][4 + j - (d - 1) / 2]));
                    }
                    const f2 xy = add2(xs, r == 0 ? add2(up[j], lo[j]) : add2(hi[j], dn[j]));
                    lap[r][j] = fma2(wd, add2(xy, zs[r][j]), lap[r][j]);
                }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                up[j] = hi[j];
                dn[j] = lo[j];
            }
            if (d < FD_NO) {
                tm_wait_ld(zp);
                tm_ready(zm);
            }
            if (d == 3) {
                v0 = ldg_stream4(vp);
                v1 = ldg_stream4(vp + 32);
            }
        }
        f2 hv[2][2];
        hv[0][0] = fma2(pack2(v0.x, v0.y), own[0][0], lap[0][0]);
        hv[0][1] = fma2(pack2(v0.z, v0.w), own[0][1], lap[0][1]);
        hv[1][0] = fma2(pack2(v1.x, v1.y), own[1][0], lap[1][0]);
        hv[1][1] = fma2(pack2(v1.z, v1.w), own[1][1], lap[1][1]);
        tm_wait_ld(sc);
        float out[8];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int i = 4 * r + 2 * j;
                const f2 o = fma2(s2, hv[r][j], pack2(-sc[i], -sc[i + 1]));
                out[i] = lo2(o);
                out[i + 1] = hi2(o);
                if (FIN) {                                // beyond the region: zero
                    out[i] = (in >> i) & 1u ? out[i] : 0.f;
                    out[i + 1] = (in >> (i + 1)) & 1u ? out[i + 1] : 0.f;
                    sum.template add<TT>(pack2(out[i], out[i + 1]), own[r][j]);
                }
            }
        tm_st8(k.tm + cb + z * 8, out);
        if (FIN && !TT && z == M && k.q == M / 4 && k.p == M / 2) *centre = (double)out[(M & 1) * 4 + (M & 3)];
        __syncwarp();
    }
    tm_wait_st();
}

// The rest of a sweep with projectors: out (columns cb, the local part) += the
// projector term, cut to the region, summed, its centre value kept.  PUB: out
// also becomes the current vector in shared memory (every reader of the old
// one is done).  ACCD: D += cd out, D in the owners' order (as the potential).
template <int M, bool TT, bool PUB, bool ACCD>
__device__ void quad_gather(const QuadCta<M>& k, uint32_t ca, uint32_t cb, QuadSums& sum, double* centre, float4* D, float cd)
{
    using G = QGeo<M>;
    const uint32_t in = quad_inside<M>(k);
    const uint2* lp = k.list + (size_t)(k.sub * G::NP + k.zi) * QD_KMAX * 32 + k.lane;
    int n = k.nvis[k.sub * G::NP + k.zi];
    uint2 next[QD_AHEAD];                                 // the next pair's entries: its list crosses the L2 meanwhile
    quad_ahead(lp, n, next);
    for (int zp = k.zi; zp < G::NP; zp += 4) {
        float nl[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) nl[i] = 0.f;
        uint2 cur[QD_AHEAD];
#pragma unroll
        for (int i = 0; i < QD_AHEAD; ++i) cur[i] = next[i];
        const uint2* lz = lp;
        const int nz = n;
        if (zp + 4 < G::NP) {
            lp += (size_t)4 * QD_KMAX * 32;
            n = k.nvis[k.sub * G::NP + zp + 4];
            quad_ahead(lp, n, next);
        }
#pragma unroll
        for (int i = 0; i < QD_AHEAD; i += 2)
            if (i < nz) {                                 // two entries' tables in flight
                const QuadTab a = quad_tables<M>(k, cur[i]), b = quad_tables<M>(k, cur[i + 1]);
                quad_visit(cur[i].y, a, nl);
                quad_visit(cur[i + 1].y, b, nl);
            }
        for (int e = QD_AHEAD; e < nz; e += 2) {          // longer lists
            const uint2 e0 = ldg_stream2(lz + e * 32), e1 = ldg_stream2(lz + (e + 1) * 32);
            const QuadTab a = quad_tables<M>(k, e0), b = quad_tables<M>(k, e1);
            quad_visit(e0.y, a, nl);
            quad_visit(e1.y, b, nl);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int z = 2 * zp + h;
            if (z >= G::S) break;                         // warp-uniform
            __syncwarp();
            float4* dz = ACCD ? D + (size_t)((k.sub * G::S + z) * 2) * 32 + k.lane : nullptr;
            float4 d0, d1;
            if (ACCD) {
                d0 = dz[0];
                d1 = dz[32];
            }
            float o[8], t[8];
            tm_ld8(k.tm + cb + z * 8, o);
            tm_ld8(k.tm + ca + z * 8, t);
            tm_wait_ld(o);
            tm_ready(t);
#pragma unroll
            for (int i = 0; i < 8; ++i) o[i] = (in >> i) & 1u ? o[i] + nl[8 * h + i] : 0.f;      // beyond the region: zero
#pragma unroll
            for (int i = 0; i < 8; i += 2) sum.template add<TT>(pack2(o[i], o[i + 1]), pack2(t[i], t[i + 1]));
            tm_st8(k.tm + cb + z * 8, o);
            if (!TT && z == M && k.q == M / 4 && k.p == M / 2) *centre = (double)o[(M & 1) * 4 + (M & 3)];
            if (ACCD) {
                dz[0] = make_float4(d0.x + cd * o[0], d0.y + cd * o[1], d0.z + cd * o[2], d0.w + cd * o[3]);
                dz[32] = make_float4(d1.x + cd * o[4], d1.y + cd * o[5], d1.z + cd * o[6], d1.w + cd * o[7]);
            }
            if (PUB && k.act) {
                float* b = k.own + z * G::PL;
                *reinterpret_cast<float4*>(b) = make_float4(o[0], o[1], o[2], o[3]);
                *reinterpret_cast<float4*>(b + G::OB) = make_float4(o[4], o[5], o[6], o[7]);
            }
            __syncwarp();
        }
    }
    tm_wait_st();
}

// One sweep of H over the region.  The local part and the inner products both
// only read the current vector, so they share a phase: on every scheduler two
// warps begin with one and two with the other, which overlaps the stencil's FP32
// and tensor-memory work with the loads of the inner products.  The gather
// follows their coefficients.  sums: out.out, out.t, t.t.
template <int M, bool TT, bool ACCD = false>
__device__ void quad_sweep(const QuadArgs& a, const QuadCta<M>& k, uint32_t ca, uint32_t cb, float s, int ncand,
                           float2 (*red)[QD_NW], double* centre, float4* D = nullptr, float cd = 0.f)
{
    QuadSums sum;
    if (a.r.nl.n_atoms > 0) {
#pragma unroll 1
        for (int ph = 0; ph < 2; ++ph) {
            if ((ph ^ k.zi) & 1) quad_stencil<M, TT, false>(a, k, ca, cb, s, sum, centre);
            else quad_dots<M>(a, k, ncand);
            __syncwarp();
        }
        quad_coefs<M>(a, k, ncand, s);
        tm_sync();                                        // the gather's planes are other warps' stencil planes
        quad_gather<M, TT, !TT, ACCD>(k, ca, cb, sum, centre, D, cd);
    } else {
        quad_stencil<M, TT, true>(a, k, ca, cb, s, sum, centre);
    }
    if (TT) {
        const float v[3] = {lo2(sum.aa) + hi2(sum.aa), lo2(sum.ab) + hi2(sum.ab), lo2(sum.ac) + hi2(sum.ac)};
        quad_warp_sums<3>(v, red);
    } else {
        const float v[2] = {lo2(sum.aa) + hi2(sum.aa), lo2(sum.ab) + hi2(sum.ab)};
        quad_warp_sums<2>(v, red);
    }
    tm_sync();
}

// The vector in columns cb becomes the current one in shared memory.
template <int M>
__device__ void quad_publish(const QuadCta<M>& k, uint32_t cb)
{
    using G = QGeo<M>;
    for (int z = k.zi; z < G::S; z += 4) {
        float v[8];
        tm_ld8(k.tm + cb + z * 8, v);
        tm_wait_ld(v);
        if (k.act) {
            float* b = k.own + z * G::PL;
            *reinterpret_cast<float4*>(b) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(b + G::OB) = make_float4(v[4], v[5], v[6], v[7]);
        }
        __syncwarp();
    }
}

// Clear the vector in shared memory and both in tensor memory.
template <int M>
__device__ void quad_clear(const QuadCta<M>& k, unsigned char* smem)
{
    using G = QGeo<M>;
    float4* t = reinterpret_cast<float4*>(smem);
    for (int i = threadIdx.x; i < G::TF / 4; i += QD_NT) t[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    const float z8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int z = k.zi; z < 2 * G::S; z += 4) tm_st8(k.tm + z * 8, z8);
    if (k.zi == 0) tm_st8(k.tm + QD_ZERO, z8);
    tm_wait_st();
}

struct QuadNode {
    int qi, qj, qk;
    const float* vwin;
    __device__ QuadNode(const RegionArgs<float>& a, long long node)
    {
        qi = (int)(node % a.g.n1);
        qj = (int)((node / a.g.n1) % a.g.n2);
        qk = (int)(node / ((long long)a.g.n1 * a.g.n2));
        vwin = a.Vp + ((size_t)qk * a.g.P2 + qj) * a.g.P1 + qi;
    }
};

// Chebyshev moments of one node (as moments_node).
template <int M>
__device__ void quad_moments_node(const QuadArgs& a, unsigned char* smem, uint32_t taddr, long long node)
{
    using G = QGeo<M>;
    __shared__ float2 red[2][QD_NW];
    __shared__ int red_i[QD_NW + 1];
    __shared__ float s_scale[3];                          // diagonal shift, 1/zeta, 2/zeta
    const bool has_nl = a.r.nl.n_atoms > 0;
    const int half = a.r.npl / 2, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    QuadCta<M> k(a, smem, taddr, has_nl, a.r.npl);
    double *s_mom = k.mom, *s_d2 = s_mom + half + 2, *s_d1 = s_d2 + half + 2;
    const QuadNode nd(a.r, node);
    if (tid == 0) {
        const double zeta = a.r.zeta[node];
        s_scale[0] = (float)(-3.0 * a.r.g.w[0] - a.r.chi[node]);
        s_scale[1] = (float)(1.0 / zeta);
        s_scale[2] = (float)(2.0 / zeta);
    }
    __syncwarp();
    quad_clear<M>(k, smem);
    tm_sync();
    quad_potential<M>(a, k, nd.vwin, s_scale[0]);
    uint32_t ca = 0, cb = G::S * 8;
    if (k.sub == M / 8 && k.zi == 0) {              // t^0 = e_q
        float e[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (k.q == M / 4 && k.p == M / 2) e[(M & 1) * 4 + (M & 3)] = 1.f;
        tm_st8(k.tm + ca + M * 8, e);
        tm_wait_st();
    }
    if (tid == 0) {
        k.t[M * G::PL + G::row(M) + M] = 1.f;
        s_mom[0] = 1.0;
    }
    int ncand = 0;
    if (has_nl) ncand = quad_setup<M>(a, k, nd.qi, nd.qj, nd.qk, red_i);
    tm_sync();
    for (int i = 0; i < half; ++i) {
        const float s = s_scale[i == 0 ? 1 : 2];
        quad_sweep<M, false>(a, k, ca, cb, s, ncand, red, &s_mom[i + 1]);
        if (warp == QD_NW - 1) {                          // one with the fewest planes
            double d[2];
            quad_cta_sums<2>(red, d);
            if (lane == 0) {
                s_d2[i + 1] = d[0];                       // t^{i+1} . t^{i+1}
                s_d1[i + 1] = d[1];                       // t^{i+1} . t^i
            }
            __syncwarp();
        }
        if (!has_nl && i + 1 < half) quad_publish<M>(k, cb);      // (the gather has published its own)
        __syncthreads();
        const uint32_t c = ca;
        ca = cb;
        cb = c;
    }
    double* out = a.r.moments + node * (long long)(a.r.npl + 1);
    for (int j = tid; j <= a.r.npl; j += QD_NT) {
        double r;
        if (j <= half) r = s_mom[j];
        else if ((j & 1) == 0) r = 2.0 * s_d2[j / 2] - s_mom[0];        // rho^{2a} = 2 t^a.t^a - rho^0
        else r = 2.0 * s_d1[(j + 1) / 2] - s_mom[1];                     // rho^{2a+1} = 2 t^{a+1}.t^a - rho^1
        out[j] = r;
        if (!(fabs(r) <= 1.0 + a.r.mom_tol)) atomicOr(a.r.err, ERR_BOUNDS);
    }
    __syncthreads();
}

// Lanczos tridiagonal of one node (as lanczos_node).
template <int M>
__device__ void quad_lanczos_node(const QuadArgs& a, unsigned char* smem, uint32_t taddr, long long node)
{
    using G = QGeo<M>;
    __shared__ float2 red[3][QD_NW];
    __shared__ int red_i[QD_NW + 1];
    __shared__ float s_alpha, s_inv, s_bprev, s_v0;
    __shared__ int s_stop, s_explicit;
    const bool has_nl = a.r.nl.n_atoms > 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    QuadCta<M> k(a, smem, taddr, has_nl, 0);
    const QuadNode nd(a.r, node);
    if (tid == 0) s_v0 = (float)(1.0 / sqrt((double)G::S * G::S * G::S));
    __syncwarp();
    quad_potential<M>(a, k, nd.vwin, a.diag);
    quad_clear<M>(k, smem);
    tm_sync();
    const float v0 = s_v0;
    uint32_t ca = 0, cb = G::S * 8;
    for (int z = k.zi; z < G::S; z += 4) {                // uniform start vector
        float e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = k.act && 4 * k.q + (i & 3) < G::S && (i < 4 || k.p < G::OD) ? v0 : 0.f;
        tm_st8(k.tm + ca + z * 8, e);
    }
    tm_wait_st();
    int ncand = 0;
    if (has_nl) ncand = quad_setup<M>(a, k, nd.qi, nd.qj, nd.qk, red_i);
    quad_publish<M>(k, ca);
    tm_sync();
    double* alpha = a.r.alpha + node * (long long)a.r.nl_cap;
    double* beta = a.r.beta + node * (long long)a.r.nl_cap;
    double bprev = 0.0, scale = 0.0;                      // thread 0 only
    for (int it = 0; it < a.r.n_lanczos; ++it) {
        // w = H v - beta_prev v_old  (columns cb hold beta_prev v_old, then w)
        quad_sweep<M, true>(a, k, ca, cb, 1.f, ncand, red, nullptr);
        // thread 0: alpha, and beta from the sweep's sums unless they cancel (as in lanczos_node)
        auto step_end = [&](double b) {
            const int stop = (it == a.r.n_lanczos - 1) || (b <= 1e-10 * scale);
            if (!stop) beta[it] = b;
            else a.r.klen[node] = it + 1;
            s_stop = stop;
            s_inv = (float)(1.0 / b);
            s_bprev = (float)b;
            bprev = b;
        };
        if (warp == 0) {
            double d[3];
            quad_cta_sums<3>(red, d);
            if (lane == 0) {
                const double al = d[1], w2 = d[0], v2 = d[2];
                alpha[it] = al;
                if (fabs(al) + bprev > scale) scale = fabs(al) + bprev;
                const double b2 = w2 - 2.0 * al * al + al * al * v2;
                s_alpha = (float)al;
                s_explicit = !(b2 > 0.01 * w2);
                if (!s_explicit) step_end(sqrt(b2));
            }
        }
        __syncthreads();
        const bool ex = s_explicit;                       // CTA-uniform
        const float alT = s_alpha;
        if (ex) {                                         // w -= alpha v ; beta = |w|
            float acc = 0.f;
            for (int z = k.zi; z < G::S; z += 4) {
                float v[8], w[8];
                tm_ld8(k.tm + ca + z * 8, v);
                tm_ld8(k.tm + cb + z * 8, w);
                tm_wait_ld(v);
                tm_ready(w);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    w[i] -= alT * v[i];
                    acc += w[i] * w[i];
                }
                tm_st8(k.tm + cb + z * 8, w);
            }
            tm_wait_st();
            const float v1[1] = {acc};
            quad_warp_sums<1>(v1, red);
            __syncthreads();
            if (warp == 0) {
                double d[1];
                quad_cta_sums<1>(red, d);
                if (lane == 0) step_end(sqrt(d[0]));
            }
            __syncthreads();
        }
        if (s_stop) break;                                // CTA-uniform
        // columns ca <- beta v (the next step's beta_prev v_old), cb and shared memory <- (w - alpha v) / beta
        const float inv = s_inv, bT = s_bprev, al2 = ex ? 0.f : alT;
        for (int z = k.zi; z < G::S; z += 4) {
            float v[8], w[8];
            tm_ld8(k.tm + ca + z * 8, v);
            tm_ld8(k.tm + cb + z * 8, w);
            tm_wait_ld(v);
            tm_ready(w);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                w[i] = (w[i] - al2 * v[i]) * inv;
                v[i] *= bT;
            }
            tm_st8(k.tm + ca + z * 8, v);
            tm_st8(k.tm + cb + z * 8, w);
            if (k.act) {
                float* b = k.own + z * G::PL;
                *reinterpret_cast<float4*>(b) = make_float4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<float4*>(b + G::OB) = make_float4(w[4], w[5], w[6], w[7]);
            }
            __syncwarp();
        }
        tm_wait_st();
        tm_sync();
        const uint32_t c = ca;
        ca = cb;
        cb = c;
    }
    __syncthreads();
}

__device__ __forceinline__ uint32_t quad_tmem_alloc(uint32_t* slot)
{
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;"
                     ::"r"((uint32_t)__cvta_generic_to_shared(slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tm_sync();
    return *slot;
}
__device__ __forceinline__ void quad_tmem_free(uint32_t taddr)
{
    tm_sync();
    if (threadIdx.x < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(taddr) : "memory");
}

// The whole register file goes to one CTA, so no other CTA that wants tensor
// memory can share its SM and the allocation never waits.
template <int M, bool LANCZOS>
__global__ void __launch_bounds__(QD_NT, 1) quad_kernel(const __grid_constant__ QuadArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_taddr;
    const uint32_t taddr = quad_tmem_alloc(&s_taddr);
    for (long long node = blockIdx.x; node < a.r.g.Nd; node += gridDim.x) {
        if (LANCZOS) quad_lanczos_node<M>(a, smem_raw, taddr, node);
        else quad_moments_node<M>(a, smem_raw, taddr, node);
    }
    quad_tmem_free(taddr);
}

// The queue of a batch (sq_queue.cuh) over systems that have quad kernels.
struct QuadQueueArgs {
    QuadArgs sys[QMAX];
    const double* V[QMAX];
    int need[QMAX];
    const QItem* items;
    int n_items;
    unsigned *next, *done;
    long long budget;
    int unset;
};

template <int M, bool LANCZOS>
__global__ void __launch_bounds__(QD_NT, 1) quad_queue_kernel(const __grid_constant__ QuadQueueArgs q)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_taddr;
    __shared__ int s_item, s_go;
    const uint32_t taddr = quad_tmem_alloc(&s_taddr);
    const int tid = threadIdx.x;
    for (;;) {
        const int it = queue_take(q.next, &s_item);
        if (it >= q.n_items) break;
        const QItem w = q.items[it];
        const QuadArgs& a = q.sys[w.sys];
        if (!LANCZOS) {
            for (long long node = w.begin; node < w.end; ++node) quad_moments_node<M>(a, smem_raw, taddr, node);
            continue;
        }
        if (w.kind == QI_VPAD) {
            for (long long t = w.begin + tid; t < w.end; t += QD_NT)
                vpad_elem<float>(q.V[w.sys], const_cast<float*>(a.r.Vp), a.r.g.n1, a.r.g.n2, a.r.g.n3, a.r.g.m, t, a.r.err);
            __syncthreads();
            if (tid == 0) {
                __threadfence();             // the slab before the count (cumulative over the CTA's writes)
                atomicAdd(q.done + w.sys, 1u);
            }
            continue;
        }
        if (tid == 0) {
            const bool ok = wait_count(q.done + w.sys, (unsigned)(q.need[w.sys] + q.unset), q.budget);
            if (!ok) atomicOr(a.r.err, ERR_TIMEOUT);
            s_go = ok;
        }
        __syncthreads();
        if (s_go) {
            for (long long node = w.begin; node < w.end; ++node) quad_lanczos_node<M>(a, smem_raw, taddr, node);
        } else {
            for (long long node = w.begin + tid; node < w.end; node += QD_NT) {
                a.r.klen[node] = 1;
                a.r.alpha[node * (long long)a.r.nl_cap] = 0.0;
            }
        }
        __syncthreads();
    }
    quad_tmem_free(taddr);
}

}  // namespace sq

#define QUAD_CASES C(7) C(8) C(9) C(10) C(11) C(12) C(13) C(14) C(15)
