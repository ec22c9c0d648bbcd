// sq_cnn_tc.cuh -- the warm-start network's 32 -> 32-channel 3^3 convolution
// (the middle layer) as an implicit GEMM on the fifth-generation tensor cores
// (tcgen05), bfloat16 operands, FP32 accumulation in tensor memory (TMEM):
//
//   z2[p][o] = b2[o] + sum_{d < 27} sum_{i < 32} W2[d][i][o] a1[p + d][i],  a2 = silu(z2)
//
// GEMM view per tile of 8 x 16 x 1 nodes: D (128 x 32) = A (128 x 864) B (864 x
// 32), row m of A = the 27 neighbour rows of node p_m (32 channels each, periodic
// wrap), B = W2 with k = d * 32 + i.  The tile's neighbourhood (10 x 18 x 3 nodes)
// is gathered into shared memory once, in an order in which every tap's A is a
// window of it: a tap is then only another start address, and one thread issues
// the tile's 54 tcgen05.mma (M = 128, N = 32, K = 16) back to back; the
// accumulator (128 lanes x 32 FP32 columns) stays in TMEM over them and four warps
// read it back with tcgen05.ld for the epilogue (bias, SiLU, stores).  The weights
// (27 x 32 x 32 bfloat16) are staged once per CTA; two CTAs per SM overlap one's
// gather with the other's MMAs and epilogue.  64^3 nodes: gathering A tap by tap
// behind a barrier each took 449 us, this takes 95 us.
//
// Operand layout (shared memory, no swizzle, K-major): 8 x 8 "core matrices" of 8
// rows x 16 bytes stored contiguously.  A: plane c of 16-byte chunks (channels 8c
// .. 8c+7) holds the 540 nodes x fastest, so 8 consecutive x are a core matrix;
// the next chunk lies LBO = 8640 bytes on, the next 8-row group (y + 1) SBO = 160
// bytes, and tap (dx, dy, dz) starts ((dz 18 + dy) 10 + dx) 16 bytes in.  B: LBO =
// 128, SBO = 512 bytes.  The second K-half of a tap starts two chunks on.
//
// Every wait on an mbarrier has an iteration limit; on expiry the kernel
// latches an error bit, stops issuing, waits (with a limit) for what it
// issued, frees its TMEM columns and returns.
#pragma once
#include "sq_cnn.cuh"

namespace sq {

constexpr int TC_M = 128;                    // nodes per tile (MMA M)
constexpr int TC_X = 8, TC_Y = 16, TC_T = 256;
constexpr int TC_TAPS = 27;
constexpr int TC_NODES = (TC_X + 2) * (TC_Y + 2) * 3;      // a tile's neighbourhood
constexpr int TC_PLANE = TC_NODES * 16;      // one 16-byte chunk of every node
constexpr int TC_BBYTES = CNN_C * CNN_C * 2; // one tap of B: 2 KB
constexpr unsigned TC_ERR_TIMEOUT = 1u;
constexpr long long TC_WAIT_LIMIT = 1ll << 26;   // mbarrier polls before giving up

// shared memory: B (27 taps), A (4 chunk planes), mbarrier, TMEM address
constexpr int TC_SMEM = TC_TAPS * TC_BBYTES + 4 * TC_PLANE + 64;

__device__ __forceinline__ uint32_t tc_smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: start >> 4 (bits 0-13), LBO >> 4 (16-29),
// SBO >> 4 (32-45), descriptor version 1 (46-47), no swizzle (61-63 = 0).
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1),
// A and B bfloat16 (7-9 = 1, 10-12 = 1), both K-major, N >> 3 (17-22),
// M >> 4 (24-28).
constexpr uint32_t TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(CNN_C >> 3) << 17) |
                              ((uint32_t)(TC_M >> 4) << 24);

__device__ __forceinline__ void tc_mbar_init(uint32_t mbar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
}

// Wait for phase `parity` of the mbarrier, at most TC_WAIT_LIMIT polls;
// false on expiry.
__device__ __forceinline__ bool tc_mbar_wait(uint32_t mbar, uint32_t parity)
{
    for (long long i = 0; i < TC_WAIT_LIMIT; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tc_mma(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(dtmem), "l"(adesc), "l"(bdesc), "r"(TC_IDESC), "r"(accumulate) : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

// z2 (may be NULL) and a2 of one layer: the forward of conv3(32 -> 32) + bias +
// SiLU on tensor cores.  256 threads per CTA, persistent over tiles.
__global__ void __launch_bounds__(TC_T) cnn_conv2_tc_kernel(CnnGrid g, const Bf16* __restrict__ x,
                                                           const Bf16* __restrict__ W,
                                                           const float* __restrict__ b,
                                                           float* __restrict__ z, Bf16* __restrict__ a,
                                                           unsigned* __restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    unsigned char* sB = tc_smem;                                  // 27 x 2 KB
    unsigned char* sA = tc_smem + TC_TAPS * TC_BBYTES;            // 4 planes
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sA + 4 * TC_PLANE);
    uint32_t* s_taddr = reinterpret_cast<uint32_t*>(mbar + 1);
    const int tid = threadIdx.x, warp = tid >> 5;

    // B: element (n = o, k = i) of tap d at core matrix (n / 8, i / 8), row n % 8, column i % 8
    for (int e = tid; e < TC_TAPS * CNN_C * CNN_C; e += TC_T) {
        const int d = e / (CNN_C * CNN_C), i = (e / CNN_C) % CNN_C, o = e % CNN_C;
        const int off = d * TC_BBYTES + ((o >> 3) * 4 + (i >> 3)) * 128 + (o & 7) * 16 + (i & 7) * 2;
        *reinterpret_cast<uint16_t*>(sB + off) = W[e].u;
    }
    if (tid == 0) {
        tc_mbar_init(tc_smem_u32(mbar));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {                                               // 32 TMEM columns: the 128 x 32 accumulator
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(tc_smem_u32(s_taddr))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = *s_taddr;
    const uint32_t sA0 = tc_smem_u32(sA), sB0 = tc_smem_u32(sB);
    uint32_t phase = 0u;
    bool ok = true;

    const long long ntiles = cnn_tiles<TC_X, TC_Y, 1>(g);
    for (long long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        const CnnTile c = cnn_tile<TC_X, TC_Y, 1>(g, tile);
        for (int i = tid; i < TC_NODES * 4; i += TC_T) {           // 16 bytes each, a node's four in adjacent lanes
            const int n = i >> 2, ch = i & 3;
            const int nx = n % (TC_X + 2), ny = (n / (TC_X + 2)) % (TC_Y + 2), nz = n / ((TC_X + 2) * (TC_Y + 2));
            const uint4 v = reinterpret_cast<const uint4*>(x + cnn_at(g, c.x + nx - 1, c.y + ny - 1, c.z + nz - 1) * CNN_C)[ch];
            *reinterpret_cast<uint4*>(sA + ch * TC_PLANE + n * 16) = v;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // A and B visible to the tensor cores
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int d = 0; d < TC_TAPS; ++d) {
                const uint32_t a0 = sA0 + (((d / 9) * (TC_Y + 2) + (d / 3) % 3) * (TC_X + 2) + d % 3) * 16;
                const uint32_t b0 = sB0 + d * TC_BBYTES;
                tc_mma(taddr, tc_desc(a0, TC_PLANE, (TC_X + 2) * 16), tc_desc(b0, 128, 512), d > 0 ? 1u : 0u);
                tc_mma(taddr, tc_desc(a0 + 2 * TC_PLANE, TC_PLANE, (TC_X + 2) * 16), tc_desc(b0 + 256, 128, 512), 1u);
            }
            tc_commit(tc_smem_u32(mbar));
            ok = tc_mbar_wait(tc_smem_u32(mbar), phase);
        }
        ok = __syncthreads_and(ok);
        phase ^= 1u;
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (warp < 4) {
            uint32_t r[32];
            const uint32_t ta = taddr + ((uint32_t)(warp * 32) << 16);   // lanes 32 warp .. 32 warp + 31
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                  "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                  "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                  "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                  "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                : "r"(ta));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            const int px = c.x + (tid & 7), py = c.y + (tid >> 3);
            if (px < g.n1 && py < g.n2) {
                const long long at = ((long long)px + (long long)g.n1 * (py + (long long)g.n2 * c.z)) * CNN_C;
#pragma unroll
                for (int o = 0; o < CNN_C; o += 8) {
                    alignas(16) Bf16 av[8];
                    alignas(16) float zv[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        zv[e] = __uint_as_float(r[o + e]) + b[o + e];
                        stv(av[e], cnn_silu(zv[e]));
                    }
                    if (z) {
                        reinterpret_cast<float4*>(z + at + o)[0] = reinterpret_cast<float4*>(zv)[0];
                        reinterpret_cast<float4*>(z + at + o)[1] = reinterpret_cast<float4*>(zv)[1];
                    }
                    *reinterpret_cast<uint4*>(a + at + o) = *reinterpret_cast<uint4*>(av);
                }
            }
        }
        // every warp has read the accumulator before the next tile's first MMA overwrites it
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
    }
    if (!ok) {
        if (tid == 0) {
            atomicOr(err, TC_ERR_TIMEOUT);
            tc_mbar_wait(tc_smem_u32(mbar), phase ^ 1u);           // what was issued, with a limit too
        }
        __syncthreads();
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(taddr) : "memory");
}

}  // namespace sq
