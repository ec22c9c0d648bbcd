// sq_cnn.cuh -- kernels of the learned SCF warm start: a 3-D convolutional
// network on the periodic grid that maps the 9^3 patch of the effective
// potential around each node to the node's density,
//
//   x0 = (V - v_shift) / v_scale
//   a1 = silu(conv5(x0; W1) + b1)      1 -> 32 channels, 5^3 kernel
//   a2 = silu(conv3(a1; W2) + b2)      32 -> 32 channels, 3^3 kernel
//   y  = conv3(a2; W3) + b3            32 -> 1 channel, 3^3 kernel
//   rho = rho_scale softplus(y)
//
// conv_k(x; W)[o](p) = sum_i sum_{d in [-r,r]^3} W[d][i][o] x[i](p + d)
// (periodic cross-correlation), its two adjoints for training, the loss
// mean((rho - rho_ref)^2)/rho_scale^2 and Adam.  Weights and activations
// are stored in T (bfloat16 or float); every sum accumulates in FP32;
// biases, pre-activations, gradients, master weights and Adam moments are
// FP32.  Layouts: activations node-major, channel fastest ([p][c]);
// weights tap-major ([d][i][o], d = (dz+r) k^2 + (dy+r) k + (dx+r)).
//
// CUDA cores but for the middle layer's forward of the bfloat16 network
// (sq_cnn_tc.cuh).  Every kernel works on tiles of nodes whose neighbourhood
// lies in shared memory and keeps a block of outputs per thread in registers, so
// the FP32 pipe bounds it rather than the loads; weight gradients are per-block
// partial sums added in block order, so everything repeats bit for bit.
#pragma once
#include <stdint.h>
#include <string.h>
#include <cuda_runtime.h>

namespace sq {

constexpr int CNN_C = 32;            // hidden channels
constexpr int CNN_NT = 256;          // threads per block
constexpr int CNN_PARTS = 96;        // blocks (partial sums) of a weight gradient, at most

// bfloat16 storage (round to nearest even from FP32; NaN stays NaN)
struct Bf16 {
    uint16_t u;
};

__host__ __device__ inline float bits_f(uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float f;
    memcpy(&f, &b, 4);
    return f;
#endif
}

__host__ __device__ inline uint32_t f_bits(float f)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    uint32_t b;
    memcpy(&b, &f, 4);
    return b;
#endif
}

__host__ __device__ inline float ldv(float v) { return v; }
__host__ __device__ inline float ldv(Bf16 v) { return bits_f((uint32_t)v.u << 16); }
__host__ __device__ inline void stv(float& d, float v) { d = v; }
__host__ __device__ inline void stv(Bf16& d, float v)
{
    uint32_t u = f_bits(v);
    if ((u & 0x7f800000u) == 0x7f800000u && (u & 0x7fffffu)) {
        d.u = (uint16_t)((u >> 16) | 0x40u);
        return;
    }
    u += 0x7fffu + ((u >> 16) & 1u);
    d.u = (uint16_t)(u >> 16);
}

__device__ inline float cnn_sigmoid(float z) { return 1.0f / (1.0f + expf(-z)); }
__device__ inline float cnn_silu(float z) { return z * cnn_sigmoid(z); }
__device__ inline float cnn_silu_grad(float z)
{
    const float s = cnn_sigmoid(z);
    return s * (1.0f + z * (1.0f - s));
}

__device__ inline int cnn_wrap(int i, int n)
{
    int r = i % n;
    return r < 0 ? r + n : r;
}

struct CnnGrid {
    int n1, n2, n3;
    long long N;
};

// x0 = (V - shift) / scale, stored in T
template <typename T>
__global__ void cnn_input_kernel(CnnGrid g, const double* __restrict__ V, double shift, double scale, T* __restrict__ x0)
{
    for (long long p = blockIdx.x * (long long)CNN_NT + threadIdx.x; p < g.N; p += (long long)gridDim.x * CNN_NT)
        stv(x0[p], (float)((V[p] - shift) / scale));
}

// A tile of TX x TY x TZ nodes and its place on the grid (ragged at the ends).
struct CnnTile {
    int x, y, z;
};
template <int TX, int TY, int TZ>
__host__ __device__ inline long long cnn_tiles(const CnnGrid& g)
{
    return (long long)((g.n1 + TX - 1) / TX) * ((g.n2 + TY - 1) / TY) * ((g.n3 + TZ - 1) / TZ);
}
template <int TX, int TY, int TZ>
__device__ inline CnnTile cnn_tile(const CnnGrid& g, long long t)
{
    const int ax = (g.n1 + TX - 1) / TX, ay = (g.n2 + TY - 1) / TY;
    return {(int)(t % ax) * TX, (int)((t / ax) % ay) * TY, (int)(t / ((long long)ax * ay)) * TZ};
}
__device__ inline long long cnn_at(const CnnGrid& g, int x, int y, int z)
{
    return (long long)cnn_wrap(x, g.n1) + (long long)g.n1 * ((long long)cnn_wrap(y, g.n2) + (long long)g.n2 * cnn_wrap(z, g.n3));
}

// First layer: z1 = b + sum_d W[d][o] x0[p + d] (5^3 taps, 32 channels), a1 =
// silu(z1) in T; z may be NULL.  A thread has 4 nodes along x and 8 channels: a
// tap costs it 2 loads of weights for 32 multiply-adds, and 5 taps share the 8
// values of x0 they read.  64^3 nodes, bfloat16: 26 us of FP32 work; a thread per
// (node, channel), one load per factor, took 720 us, this takes 65 us.
constexpr int C1_X = 8, C1_Y = 8, C1_Z = 4;
template <typename T>
__global__ void __launch_bounds__(CNN_NT) cnn_conv1_kernel(CnnGrid g, const T* __restrict__ x0, const T* __restrict__ W,
                                                           const float* __restrict__ b, float* __restrict__ z,
                                                           T* __restrict__ a)
{
    constexpr int PX = C1_X + 4, PY = C1_Y + 4, PZ = C1_Z + 4;
    __shared__ __align__(16) float sx[PX * PY * PZ];
    __shared__ __align__(16) float sw[125 * CNN_C];
    for (int i = threadIdx.x; i < 125 * CNN_C; i += CNN_NT) sw[i] = ldv(W[i]);
    const int cg = threadIdx.x & 3, nq = threadIdx.x >> 2;       // 8 channels, quad of nodes
    const int lx = (nq & 1) * 4, ly = (nq >> 1) & 7, lz = nq >> 4;
    float bias[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) bias[o] = b[8 * cg + o];
    const long long nt = cnn_tiles<C1_X, C1_Y, C1_Z>(g);
    for (long long t = blockIdx.x; t < nt; t += gridDim.x) {
        const CnnTile c = cnn_tile<C1_X, C1_Y, C1_Z>(g, t);
        __syncthreads();
        for (int i = threadIdx.x; i < PX * PY * PZ; i += CNN_NT)
            sx[i] = ldv(x0[cnn_at(g, c.x + i % PX - 2, c.y + (i / PX) % PY - 2, c.z + i / (PX * PY) - 2)]);
        __syncthreads();
        float acc[4][8];
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int o = 0; o < 8; ++o) acc[n][o] = 0.0f;
        for (int dz = 0; dz < 5; ++dz)
            for (int dy = 0; dy < 5; ++dy) {
                const float4* row = reinterpret_cast<const float4*>(sx + ((lz + dz) * PY + ly + dy) * PX + lx);
                const float4 u = row[0], v = row[1];
                const float xs[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
                const float4* w4 = reinterpret_cast<const float4*>(sw + (dz * 5 + dy) * 5 * CNN_C + 8 * cg);
#pragma unroll
                for (int dx = 0; dx < 5; ++dx) {
                    const float4 p = w4[dx * (CNN_C / 4)], q = w4[dx * (CNN_C / 4) + 1];
                    const float w[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int n = 0; n < 4; ++n)
#pragma unroll
                        for (int o = 0; o < 8; ++o) acc[n][o] += w[o] * xs[n + dx];
                }
            }
        const int py = c.y + ly, pz = c.z + lz;
        if (py < g.n2 && pz < g.n3)
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                const int px = c.x + lx + n;
                if (px >= g.n1) break;
                const long long at = ((long long)px + (long long)g.n1 * (py + (long long)g.n2 * pz)) * CNN_C + 8 * cg;
                alignas(16) T av[8];
                alignas(16) float zv[8];
#pragma unroll
                for (int o = 0; o < 8; ++o) {
                    zv[o] = acc[n][o] + bias[o];
                    stv(av[o], cnn_silu(zv[o]));
                }
                if (z) {
                    reinterpret_cast<float4*>(z + at)[0] = reinterpret_cast<float4*>(zv)[0];
                    reinterpret_cast<float4*>(z + at)[1] = reinterpret_cast<float4*>(zv)[1];
                }
#pragma unroll
                for (int h = 0; h < (int)(8 * sizeof(T) / 16); ++h)
                    reinterpret_cast<uint4*>(a + at)[h] = reinterpret_cast<uint4*>(av)[h];
            }
    }
}

// 32 -> 32 channel 3^3 convolution on CUDA cores, both ways:
//   forward (BWD = false): z = b + sum_d sum_i W[d][i][o] x[p + d][i], a = silu(z)
//   data gradient (BWD = true): gx[p][i] = (sum_d sum_o W[d][i][o] gz[p - d][o]) silu'(zx[p][i])
// In both a tap is a 32 x 32 matrix applied to the neighbour's 32 values.  A
// thread has 4 nodes along x and 8 of the 32 results, summed per (dz, dy); per input channel and (dz,
// dy) it reads 6 neighbours and 3 x 8 weights for 96 multiply-adds.  Neighbours
// in shared memory by channel, weights per (dz, dy).  Data
// gradient on 16^3 nodes (32 blocks of work for 152 SMs, each a chain of nine
// weight tiles): a thread per (node, channel) took 237 us, this takes 59 us.
constexpr int C2_X = 8, C2_Y = 8, C2_Z = 2, C2_T = 128;
constexpr int C2_PX = 12, C2_PLANE = C2_PX * (C2_Y + 2) * (C2_Z + 2) + 4;      // +4: channels in other banks
constexpr size_t C2_SMEM = ((size_t)CNN_C * C2_PLANE + 3 * CNN_C * CNN_C) * sizeof(float);

template <typename TX, typename T, bool BWD>
__global__ void __launch_bounds__(C2_T) cnn_conv2_kernel(CnnGrid g, const TX* __restrict__ x, const T* __restrict__ W,
                                                         const float* __restrict__ b, const float* __restrict__ zx,
                                                         float* __restrict__ z, T* __restrict__ a)
{
    extern __shared__ __align__(16) float csm[];
    float* sx = csm;                                     // [channel][plane][row][12]
    float* sw = csm + CNN_C * C2_PLANE;                  // [dx][in][out] of one (dz, dy)
    const int cg = threadIdx.x & 3, nq = threadIdx.x >> 2;
    const int lx = (nq & 1) * 4, ly = (nq >> 1) & 7, lz = nq >> 4;
    constexpr int NODES = (C2_X + 2) * (C2_Y + 2) * (C2_Z + 2);
    const long long nt = cnn_tiles<C2_X, C2_Y, C2_Z>(g);
    for (long long t = blockIdx.x; t < nt; t += gridDim.x) {
        const CnnTile c = cnn_tile<C2_X, C2_Y, C2_Z>(g, t);
        __syncthreads();
        for (int i = threadIdx.x; i < NODES * 8; i += C2_T) {      // 4 channels of a neighbour
            const int n = i >> 3, ch = (i & 7) * 4;
            const int nx = n % (C2_X + 2), ny = (n / (C2_X + 2)) % (C2_Y + 2), nz = n / ((C2_X + 2) * (C2_Y + 2));
            const TX* src = x + cnn_at(g, c.x + nx - 1, c.y + ny - 1, c.z + nz - 1) * CNN_C + ch;
#pragma unroll
            for (int e = 0; e < 4; ++e) sx[(ch + e) * C2_PLANE + (nz * (C2_Y + 2) + ny) * C2_PX + nx] = ldv(src[e]);
        }
        float acc[4][8], tap[4][8];
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int o = 0; o < 8; ++o) acc[n][o] = 0.0f;
        for (int dzy = 0; dzy < 9; ++dzy) {
            __syncthreads();
            for (int i = threadIdx.x; i < 3 * CNN_C * CNN_C; i += C2_T) {
                const int dx = i >> 10, in = (i >> 5) & 31, out = i & 31;
                // the data gradient reads p - d: the mirrored tap, its matrix transposed
                const int d = BWD ? 26 - (dzy * 3 + dx) : dzy * 3 + dx;
                sw[i] = BWD ? ldv(W[((size_t)d * CNN_C + out) * CNN_C + in]) : ldv(W[((size_t)d * CNN_C + in) * CNN_C + out]);
            }
            __syncthreads();
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll
                for (int o = 0; o < 8; ++o) tap[n][o] = 0.0f;
            const float* row = sx + ((lz + dzy / 3) * (C2_Y + 2) + ly + dzy % 3) * C2_PX + lx;
            const float4* w4 = reinterpret_cast<const float4*>(sw + 8 * cg);
#pragma unroll 4
            for (int in = 0; in < CNN_C; ++in) {
                const float4 u = *reinterpret_cast<const float4*>(row + in * C2_PLANE);
                const float2 v = *reinterpret_cast<const float2*>(row + in * C2_PLANE + 4);
                const float xs[6] = {u.x, u.y, u.z, u.w, v.x, v.y};
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    const float4 p = w4[(dx * CNN_C + in) * (CNN_C / 4)], q = w4[(dx * CNN_C + in) * (CNN_C / 4) + 1];
                    const float w[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int n = 0; n < 4; ++n)
#pragma unroll
                        for (int o = 0; o < 8; ++o) tap[n][o] += w[o] * xs[n + dx];
                }
            }
#pragma unroll
            for (int n = 0; n < 4; ++n)
#pragma unroll
                for (int o = 0; o < 8; ++o) acc[n][o] += tap[n][o];
        }
        const int py = c.y + ly, pz = c.z + lz;
        if (py < g.n2 && pz < g.n3)
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                const int px = c.x + lx + n;
                if (px >= g.n1) break;
                const long long at = ((long long)px + (long long)g.n1 * (py + (long long)g.n2 * pz)) * CNN_C + 8 * cg;
#pragma unroll
                for (int o = 0; o < 8; ++o) {
                    if (BWD) {
                        z[at + o] = acc[n][o] * cnn_silu_grad(zx[at + o]);
                    } else {
                        const float zz = acc[n][o] + b[8 * cg + o];
                        if (z) z[at + o] = zz;
                        stv(a[at + o], cnn_silu(zz));
                    }
                }
            }
    }
}

// Output layer: y[p] = b3 + sum_d sum_i W3[d][i] a2[p + d][i]; rho = rs softplus(y)
// (y may be NULL).  A thread per node, the tile's a2 in shared memory at a node
// pitch that is an odd multiple of 16 bytes.  64^3 nodes, bfloat16: 410 us with
// every neighbour read from global memory, 48 us so.
constexpr int C3_X = 8, C3_Y = 8, C3_Z = 4;
template <typename T>
constexpr int c3_pitch() { return (int)(CNN_C * sizeof(T) / 16 + 1) * 16; }
template <typename T>
constexpr size_t c3_smem() { return (size_t)(C3_X + 2) * (C3_Y + 2) * (C3_Z + 2) * c3_pitch<T>() + 27 * CNN_C * sizeof(float); }

template <typename T>
__global__ void __launch_bounds__(CNN_NT) cnn_out_fwd_kernel(CnnGrid g, const T* __restrict__ a2,
                                                             const T* __restrict__ W3, const float* __restrict__ b3,
                                                             double rho_scale, float* __restrict__ y,
                                                             double* __restrict__ rho)
{
    extern __shared__ __align__(16) unsigned char osm[];
    constexpr int NODES = (C3_X + 2) * (C3_Y + 2) * (C3_Z + 2), PITCH = c3_pitch<T>(), V = CNN_C * sizeof(T) / 16;
    float* sw = reinterpret_cast<float*>(osm + (size_t)NODES * PITCH);
    for (int i = threadIdx.x; i < 27 * CNN_C; i += CNN_NT) sw[i] = ldv(W3[i]);
    const int lx = threadIdx.x & 7, ly = (threadIdx.x >> 3) & 7, lz = threadIdx.x >> 6;
    const long long nt = cnn_tiles<C3_X, C3_Y, C3_Z>(g);
    for (long long t = blockIdx.x; t < nt; t += gridDim.x) {
        const CnnTile c = cnn_tile<C3_X, C3_Y, C3_Z>(g, t);
        __syncthreads();
        for (int i = threadIdx.x; i < NODES * V; i += CNN_NT) {
            const int n = i / V, v = i % V;
            const int nx = n % (C3_X + 2), ny = (n / (C3_X + 2)) % (C3_Y + 2), nz = n / ((C3_X + 2) * (C3_Y + 2));
            *reinterpret_cast<uint4*>(osm + n * PITCH + v * 16) =
                reinterpret_cast<const uint4*>(a2 + cnn_at(g, c.x + nx - 1, c.y + ny - 1, c.z + nz - 1) * CNN_C)[v];
        }
        __syncthreads();
        const int px = c.x + lx, py = c.y + ly, pz = c.z + lz;
        if (px < g.n1 && py < g.n2 && pz < g.n3) {
            float acc = 0.0f;
            for (int d = 0; d < 27; ++d) {
                float tap = 0.0f;
                const unsigned char* src =
                    osm + (((lz + d / 9) * (C3_Y + 2) + ly + (d / 3) % 3) * (C3_X + 2) + lx + d % 3) * PITCH;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    alignas(16) T xs[16 / sizeof(T)];
                    *reinterpret_cast<uint4*>(xs) = *reinterpret_cast<const uint4*>(src + v * 16);
                    const float* w = sw + d * CNN_C + v * (16 / sizeof(T));
#pragma unroll
                    for (int e = 0; e < (int)(16 / sizeof(T)); ++e) tap += w[e] * ldv(xs[e]);
                }
                acc += tap;
            }
            const long long p = (long long)px + (long long)g.n1 * (py + (long long)g.n2 * pz);
            const float yy = acc + b3[0];
            if (y) y[p] = yy;
            const float sp = fmaxf(yy, 0.0f) + log1pf(expf(-fabsf(yy)));
            rho[p] = rho_scale * (double)sp;
        }
    }
}

// Loss partials and dL/dy: diff = rho - ref, part[block] = sum diff^2 (tree
// in shared memory), gy = 2 diff / (N rs^2) * rs * sigmoid(y).
__global__ void __launch_bounds__(CNN_NT) cnn_loss_kernel(CnnGrid g, const double* __restrict__ rho,
                                                          const double* __restrict__ ref, const float* __restrict__ y,
                                                          double rho_scale, float* __restrict__ gy,
                                                          double* __restrict__ part)
{
    __shared__ double s[CNN_NT];
    double acc = 0.0;
    const double cg = 2.0 / ((double)g.N * rho_scale);
    for (long long p = blockIdx.x * (long long)CNN_NT + threadIdx.x; p < g.N; p += (long long)gridDim.x * CNN_NT) {
        const double dlt = rho[p] - ref[p];
        acc += dlt * dlt;
        gy[p] = (float)(cg * dlt) * cnn_sigmoid(y[p]);
    }
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int w = CNN_NT / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

// part[block] = sum of rho over the block's nodes (tree in shared memory).
__global__ void __launch_bounds__(CNN_NT) cnn_sum_kernel(CnnGrid g, const double* __restrict__ rho,
                                                         double* __restrict__ part)
{
    __shared__ double s[CNN_NT];
    double acc = 0.0;
    for (long long p = blockIdx.x * (long long)CNN_NT + threadIdx.x; p < g.N; p += (long long)gridDim.x * CNN_NT)
        acc += rho[p];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int w = CNN_NT / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = s[0];
}

// out[0] = (sum_b part[b]) / (N rs^2), in block order (one thread).
__global__ void cnn_loss_sum_kernel(const double* __restrict__ part, int nb, double norm, double* __restrict__ out)
{
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    double s = 0.0;
    for (int b = 0; b < nb; ++b) s += part[b];
    out[0] = s * norm;
}

// Data gradient through the output layer: gz2[p][c] = (sum_d W3[d][c] gy[p - d])
// silu'(z2[p][c]).  A lane per channel with its 27 weights in registers, a warp
// per row of 8 nodes, gy of the tile in shared memory.
template <typename T>
__global__ void __launch_bounds__(CNN_NT) cnn_out_bwd_kernel(CnnGrid g, const float* __restrict__ gy,
                                                             const T* __restrict__ W3, const float* __restrict__ z2,
                                                             float* __restrict__ gz2)
{
    constexpr int X = 8, Y = 8, Z = 2, PX = 12, PY = Y + 2, PZ = Z + 2;
    __shared__ __align__(16) float sg[PX * PY * PZ];
    const int c = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float w[27];
#pragma unroll
    for (int d = 0; d < 27; ++d) w[d] = ldv(W3[(26 - d) * CNN_C + c]);       // gy[p - d]: the mirrored tap
    const long long nt = cnn_tiles<X, Y, Z>(g);
    for (long long t = blockIdx.x; t < nt; t += gridDim.x) {
        const CnnTile tl = cnn_tile<X, Y, Z>(g, t);
        __syncthreads();
        for (int i = threadIdx.x; i < PX * PY * PZ; i += CNN_NT) {
            const int nx = i % PX;
            if (nx < X + 2) sg[i] = gy[cnn_at(g, tl.x + nx - 1, tl.y + (i / PX) % PY - 1, tl.z + i / (PX * PY) - 1)];
        }
        __syncthreads();
        for (int r = warp; r < Y * Z; r += CNN_NT / 32) {
            const int ly = r % Y, lz = r / Y;
            float acc[X];
#pragma unroll
            for (int n = 0; n < X; ++n) acc[n] = 0.0f;
#pragma unroll
            for (int dzy = 0; dzy < 9; ++dzy) {
                const float* row = sg + ((lz + dzy / 3) * PY + ly + dzy % 3) * PX;
                float v[X + 2];
#pragma unroll
                for (int n = 0; n < X + 2; ++n) v[n] = row[n];
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                    for (int n = 0; n < X; ++n) acc[n] += w[3 * dzy + dx] * v[n + dx];
            }
            const int py = tl.y + ly, pz = tl.z + lz;
            if (py < g.n2 && pz < g.n3)
#pragma unroll
                for (int n = 0; n < X; ++n)
                    if (tl.x + n < g.n1) {
                        const long long at = ((long long)(tl.x + n) + (long long)g.n1 * (py + (long long)g.n2 * pz)) * CNN_C + c;
                        gz2[at] = acc[n] * cnn_silu_grad(z2[at]);
                    }
        }
    }
}

// Weight-gradient partials of block (part, slab): the sum over the block's tiles
// of G[p][o] A[p + d][i] into part[block][d][i][o], for the taps of the slab; the
// extra tap K^3 is the bias (A = 1, input 0).  Tiles of 8 x 8 x 2 nodes, A with
// its neighbours and G in shared memory (zero beyond the grid); rows of 8 nodes
// along x share the loads of A between the taps dx and those of G between dy.
// Every tile's sums are added to part by themselves: FP32 chains of 128 nodes and
// then of tiles (171 at 128^3), not of all the block's nodes (21,888 there).  The
// additions are reductions that nothing waits for (a gradient at 64^3, one sample:
// 1.86 ms with one chain per block, 1.99 with the sums read back, 1.88 so); one
// thread's reductions of one address keep their order.
// 16^3 nodes: a block per (4096 nodes, tap), each node in turn, took 464 us for the
// middle layer, 374 for the last and 898 for the first; these take 21, 20 and 11.
constexpr int WG_X = 8, WG_Y = 8, WG_Z = 2;

// Middle layer (32 x 32 per tap): slab = dz, a thread has one input, four outputs and the slab's 9 taps.
constexpr size_t WG2_SMEM =
    ((size_t)(WG_X + 2) * (WG_Y + 2) * WG_Z * (CNN_C + 1) + (size_t)WG_X * WG_Y * WG_Z * CNN_C) * sizeof(float) + 16;
template <typename T>
__global__ void __launch_bounds__(CNN_NT) cnn_wgrad2_kernel(CnnGrid g, const float* __restrict__ G,
                                                            const T* __restrict__ A, float* __restrict__ part)
{
    extern __shared__ __align__(16) float wsm2[];
    constexpr int PX = WG_X + 2, PY = WG_Y + 2, NODES = PX * PY * WG_Z, OWN = WG_X * WG_Y * WG_Z;
    float* sG = wsm2;                                    // [node][32]
    float* sA = wsm2 + OWN * CNN_C;                      // [node][33]
    const int in = threadIdx.x & 31, oq = threadIdx.x >> 5;
    const int dz = (int)blockIdx.y - 1;
    float* out = part + (size_t)blockIdx.x * 28 * CNN_C * CNN_C;
    const long long nt = cnn_tiles<WG_X, WG_Y, WG_Z>(g);
    for (long long t = blockIdx.x; t < nt; t += gridDim.x) {
        const CnnTile c = cnn_tile<WG_X, WG_Y, WG_Z>(g, t);
        __syncthreads();
        for (int i = threadIdx.x; i < NODES * CNN_C; i += CNN_NT) {
            const int n = i >> 5, ch = i & 31;
            const int nx = n % PX, ny = (n / PX) % PY, nz = n / (PX * PY);
            sA[n * (CNN_C + 1) + ch] = ldv(A[cnn_at(g, c.x + nx - 1, c.y + ny - 1, c.z + nz + dz) * CNN_C + ch]);
        }
        for (int i = threadIdx.x; i < OWN * CNN_C; i += CNN_NT) {
            const int n = i >> 5, ch = i & 31;
            const int px = c.x + n % WG_X, py = c.y + (n / WG_X) % WG_Y, pz = c.z + n / (WG_X * WG_Y);
            sG[i] = px < g.n1 && py < g.n2 && pz < g.n3
                        ? G[((long long)px + (long long)g.n1 * (py + (long long)g.n2 * pz)) * CNN_C + ch] : 0.0f;
        }
        __syncthreads();
        float acc[9][4], bias[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int d = 0; d < 9; ++d)
#pragma unroll
            for (int o = 0; o < 4; ++o) acc[d][o] = 0.0f;
        for (int r = 0; r < WG_Y * WG_Z; ++r) {
            const int ly = r % WG_Y, lz = r / WG_Y;
            float4 gv[WG_X];
#pragma unroll
            for (int n = 0; n < WG_X; ++n) gv[n] = *reinterpret_cast<const float4*>(sG + (r * WG_X + n) * CNN_C + 4 * oq);
            if (dz == 0 && in == 0)
#pragma unroll
                for (int n = 0; n < WG_X; ++n) {
                    bias[0] += gv[n].x;
                    bias[1] += gv[n].y;
                    bias[2] += gv[n].z;
                    bias[3] += gv[n].w;
                }
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const float* row = sA + ((lz * PY + ly + dy) * PX) * (CNN_C + 1) + in;
                float v[WG_X + 2];
#pragma unroll
                for (int n = 0; n < WG_X + 2; ++n) v[n] = row[n * (CNN_C + 1)];
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                    for (int n = 0; n < WG_X; ++n) {
                        acc[3 * dy + dx][0] += gv[n].x * v[n + dx];
                        acc[3 * dy + dx][1] += gv[n].y * v[n + dx];
                        acc[3 * dy + dx][2] += gv[n].z * v[n + dx];
                        acc[3 * dy + dx][3] += gv[n].w * v[n + dx];
                    }
            }
        }
        const bool first = t == blockIdx.x;
        auto add = [&](float* to, const float (&v)[4]) {
            if (first) *reinterpret_cast<float4*>(to) = make_float4(v[0], v[1], v[2], v[3]);
            else asm volatile("red.global.add.v4.f32 [%0], {%1,%2,%3,%4};"
                              ::"l"(to), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
        };
#pragma unroll
        for (int d = 0; d < 9; ++d) add(out + ((size_t)((dz + 1) * 9 + d) * CNN_C + in) * CNN_C + 4 * oq, acc[d]);
        if (dz == 0 && in == 0) add(out + (size_t)27 * CNN_C * CNN_C + 4 * oq, bias);
    }
}

// First layer (1 -> 32, 5^3 taps): a lane per output, a warp per group of (dz, dy) rows of taps.
template <typename T>
__global__ void __launch_bounds__(CNN_NT) cnn_wgrad1_kernel(CnnGrid g, const float* __restrict__ G,
                                                            const T* __restrict__ A, float* __restrict__ part)
{
    constexpr int PX = WG_X + 4, PY = WG_Y + 4, PZ = WG_Z + 4, OWN = WG_X * WG_Y * WG_Z, NG = CNN_NT / 32;
    __shared__ __align__(16) float sG[OWN * CNN_C], sA[PX * PY * PZ];
    const int o = threadIdx.x & 31, grp = threadIdx.x >> 5;
    float* out = part + (size_t)blockIdx.x * 126 * CNN_C;
    const long long nt = cnn_tiles<WG_X, WG_Y, WG_Z>(g);
    for (long long t = blockIdx.x; t < nt; t += gridDim.x) {
        const CnnTile c = cnn_tile<WG_X, WG_Y, WG_Z>(g, t);
        __syncthreads();
        for (int i = threadIdx.x; i < PX * PY * PZ; i += CNN_NT)
            sA[i] = ldv(A[cnn_at(g, c.x + i % PX - 2, c.y + (i / PX) % PY - 2, c.z + i / (PX * PY) - 2)]);
        for (int i = threadIdx.x; i < OWN * CNN_C; i += CNN_NT) {
            const int n = i >> 5, ch = i & 31;
            const int px = c.x + n % WG_X, py = c.y + (n / WG_X) % WG_Y, pz = c.z + n / (WG_X * WG_Y);
            sG[i] = px < g.n1 && py < g.n2 && pz < g.n3
                        ? G[((long long)px + (long long)g.n1 * (py + (long long)g.n2 * pz)) * CNN_C + ch] : 0.0f;
        }
        __syncthreads();
        float acc[4][5], bias = 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int d = 0; d < 5; ++d) acc[i][d] = 0.0f;
        for (int r = 0; r < WG_Y * WG_Z; ++r) {
            const int ly = r % WG_Y, lz = r / WG_Y;
            float gv[WG_X];
#pragma unroll
            for (int n = 0; n < WG_X; ++n) gv[n] = sG[(r * WG_X + n) * CNN_C + o];
            if (grp == 0)
#pragma unroll
                for (int n = 0; n < WG_X; ++n) bias += gv[n];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int dzy = grp + NG * i;
                if (dzy < 25) {
                    const float* row = sA + ((lz + dzy / 5) * PY + ly + dzy % 5) * PX;
                    float v[WG_X + 4];
#pragma unroll
                    for (int n = 0; n < WG_X + 4; ++n) v[n] = row[n];
#pragma unroll
                    for (int dx = 0; dx < 5; ++dx)
#pragma unroll
                        for (int n = 0; n < WG_X; ++n) acc[i][dx] += gv[n] * v[n + dx];
                }
            }
        }
        const bool first = t == blockIdx.x;
        auto add = [&](float* to, float v) {
            if (first) *to = v;
            else asm volatile("red.global.add.f32 [%0], %1;" ::"l"(to), "f"(v) : "memory");
        };
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (grp + NG * i < 25)
#pragma unroll
                for (int dx = 0; dx < 5; ++dx) add(out + ((grp + NG * i) * 5 + dx) * CNN_C + o, acc[i][dx]);
        if (grp == 0) add(out + 125 * CNN_C + o, bias);
    }
}

// Output layer (32 -> 1, 3^3 taps): a lane per input, a warp per row of taps; the
// bias is the sum of G (input 0 of the extra tap).
template <typename T>
__global__ void __launch_bounds__(CNN_NT) cnn_wgrad3_kernel(CnnGrid g, const float* __restrict__ G,
                                                            const T* __restrict__ A, float* __restrict__ part)
{
    extern __shared__ __align__(16) float wsm3[];
    constexpr int PX = WG_X + 2, PY = WG_Y + 2, PZ = WG_Z + 2, OWN = WG_X * WG_Y * WG_Z, NG = CNN_NT / 32;
    float* sA = wsm3;                                    // [node][32]
    float* sG = wsm3 + PX * PY * PZ * CNN_C;
    const int in = threadIdx.x & 31, grp = threadIdx.x >> 5;
    float* out = part + (size_t)blockIdx.x * 28 * CNN_C;
    const long long nt = cnn_tiles<WG_X, WG_Y, WG_Z>(g);
    for (long long t = blockIdx.x; t < nt; t += gridDim.x) {
        const CnnTile c = cnn_tile<WG_X, WG_Y, WG_Z>(g, t);
        __syncthreads();
        for (int i = threadIdx.x; i < PX * PY * PZ * CNN_C; i += CNN_NT) {
            const int n = i >> 5, ch = i & 31;
            const int nx = n % PX, ny = (n / PX) % PY, nz = n / (PX * PY);
            sA[i] = ldv(A[cnn_at(g, c.x + nx - 1, c.y + ny - 1, c.z + nz - 1) * CNN_C + ch]);
        }
        for (int n = threadIdx.x; n < OWN; n += CNN_NT) {
            const int px = c.x + n % WG_X, py = c.y + (n / WG_X) % WG_Y, pz = c.z + n / (WG_X * WG_Y);
            sG[n] = px < g.n1 && py < g.n2 && pz < g.n3 ? G[(long long)px + (long long)g.n1 * (py + (long long)g.n2 * pz)] : 0.0f;
        }
        __syncthreads();
        float acc[2][3] = {{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}}, bias = 0.0f;
        for (int r = 0; r < WG_Y * WG_Z; ++r) {
            const int ly = r % WG_Y, lz = r / WG_Y;
            float gv[WG_X];
#pragma unroll
            for (int n = 0; n < WG_X; ++n) gv[n] = sG[r * WG_X + n];
            if (grp == 0)
#pragma unroll
                for (int n = 0; n < WG_X; ++n) bias += gv[n];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int dzy = grp + NG * i;
                if (dzy < 9) {
                    const float* row = sA + ((lz + dzy / 3) * PY + ly + dzy % 3) * PX * CNN_C + in;
                    float v[WG_X + 2];
#pragma unroll
                    for (int n = 0; n < WG_X + 2; ++n) v[n] = row[n * CNN_C];
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                        for (int n = 0; n < WG_X; ++n) acc[i][dx] += gv[n] * v[n + dx];
                }
            }
        }
        const bool first = t == blockIdx.x;
        auto add = [&](float* to, float v) {
            if (first) *to = v;
            else asm volatile("red.global.add.f32 [%0], %1;" ::"l"(to), "f"(v) : "memory");
        };
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (grp + NG * i < 9)
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) add(out + ((grp + NG * i) * 3 + dx) * CNN_C + in, acc[i][dx]);
        if (grp == 0) add(out + 27 * CNN_C + in, in == 0 ? bias : 0.0f);
    }
}
constexpr size_t WG3_SMEM = ((size_t)(WG_X + 2) * (WG_Y + 2) * (WG_Z + 2) * CNN_C + WG_X * WG_Y * WG_Z) * sizeof(float);

// grad[d][e] = sum over blocks (in order) of part[block][d][e], for the
// TAPS + 1 taps of one layer; the bias (tap TAPS) keeps its first CO entries.
__global__ void cnn_wgrad_sum_kernel(const float* __restrict__ part, int nchunk, int taps1, int nout, int co,
                                     float* __restrict__ gw, float* __restrict__ gb, int accumulate)
{
    const long long n = (long long)taps1 * nout;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        float s = 0.0f;
        for (int c = 0; c < nchunk; ++c) s += part[(size_t)c * n + t];
        const long long d = t / nout;
        const int e = (int)(t % nout);
        if (d < taps1 - 1) {
            gw[t] = accumulate ? gw[t] + s : s;
        } else if (e < co) {
            gb[e] = accumulate ? gb[e] + s : s;
        }
    }
}

// Adam on the FP32 master weights (flat), then the compute copy in T:
// m = b1 m + (1-b1) g s, v = b2 v + (1-b2) (g s)^2, w -= lr (m c1) / (sqrt(v c2) + eps)
// with s the gradient scale and c1, c2 the bias corrections 1/(1 - b^t).
__global__ void cnn_adam_kernel(long long n, float* __restrict__ w, const float* __restrict__ gr,
                                float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2, float eps,
                                float c1, float c2, float gscale)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const float gg = gr[t] * gscale;
        const float mm = b1 * m[t] + (1.0f - b1) * gg;
        const float vv = b2 * v[t] + (1.0f - b2) * gg * gg;
        m[t] = mm;
        v[t] = vv;
        w[t] -= lr * (mm * c1) / (sqrtf(vv * c2) + eps);
    }
}

// Compute copies of the weights: dst[t] = T(src[t]).
template <typename T>
__global__ void cnn_cast_kernel(long long n, const float* __restrict__ src, T* __restrict__ dst)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
        stv(dst[t], src[t]);
}

}  // namespace sq
