// tcgen05, TMEM and mbarrier helpers shared by the tensor-core kernels.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace tbsci {

// x = sum of NP BF16 values, each the rounded rest of the ones before
template <int NP>
__device__ __forceinline__ void bf16_planes(float x, uint32_t (&h)[NP]) {
#pragma unroll
    for (int s = 0; s < NP; ++s) {
        const __nv_bfloat16 b = __float2bfloat16_rn(x);
        h[s] = __bfloat16_as_ushort(b);
        if (s + 1 < NP) {
            const float r = x - __bfloat162float(b);
            x = isfinite(r) ? r : 0.f;  // infinities and NaN lie in the first plane
        }
    }
}

__device__ __forceinline__ uint32_t su32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Bounded wait on an mbarrier phase; gives up when another thread did (abort flag).
__device__ __forceinline__ bool mb_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 63) == 63 && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
__device__ __forceinline__ void mb_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mb_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory operand descriptor: start, leading / stride byte offsets, swizzle (2: 128 B, 4: 64 B)
__device__ __forceinline__ uint64_t op_desc(uint32_t addr, uint32_t lbo, uint32_t sbo, uint32_t swizzle) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46) | ((uint64_t)swizzle << 61);
}
// instruction descriptor: D FP32, A and B BF16, A K-major, B K- or MN-major, M = 128
__host__ __device__ constexpr uint32_t inst_desc(int n, bool b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(128 >> 4) << 24);
}

// One lane of the (converged) issuing warp. The operands of tcgen05.mma live in uniform
// registers: a warp-uniform value (`uni`) outside and immediate offsets inside keep the
// issue at a few instructions per product; with per-thread descriptors each took 150
// cycles, five times the product itself.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ uint32_t uni(uint32_t x) { return __reduce_max_sync(0xffffffffu, x); }

// D += A B: A plane from shared memory, kept in the collector over a run of products (R: 0 single, 1 first, 2 inner, 3 last)
template <int R>
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t keep) {
    if (R == 0)
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
                     "l"(a), "l"(b), "r"(idesc), "r"(keep)
                     : "memory");
    else if (R == 1)
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], %1, %2, %3, p;\n}" ::"r"(d),
            "l"(a), "l"(b), "r"(idesc), "r"(keep)
            : "memory");
    else if (R == 2)
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%0], %1, %2, %3, p;\n}" ::"r"(d),
            "l"(a), "l"(b), "r"(idesc), "r"(keep)
            : "memory");
    else
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%0], %1, %2, %3, p;\n}" ::"r"(d),
            "l"(a), "l"(b), "r"(idesc), "r"(keep)
            : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// keeps uses of r behind the wait for its load
__device__ __forceinline__ void pin16(uint32_t (&r)[16]) {
    asm volatile(""
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
}

// shapes of the alpha-beta kernels
constexpr int kAbTile = 64;       // beta columns of a tile
constexpr int kAbDrain = 512;     // draining threads (16 warps)
constexpr int kAbThreads = 640;   // and 3 staging warps and an MMA warp
constexpr int kAbMaxK = 80;       // alpha terms of a row, padded to 16 (norb <= 16: at most 65)
constexpr int kPiece = 4;         // slots that one thread sums (lists are cut into pieces)

// Gathers the columns 64 t .. 64 t + 63 of NP planes [la][lbp] of c, rows sJa[0 .. Kp - 1],
// into stage `dst` by one warp: MN-major operand planes of Kp rows of 128 bytes, 128-byte swizzle.
template <int NP>
__device__ __forceinline__ void gather_tile(const __nv_bfloat16 *C, size_t plane, int64_t lbp, const int *sJa, int Kp, int t,
                                            uint32_t dst0) {
    const int lane = threadIdx.x & 31, c16 = lane & 7, r = lane >> 3;
    const __nv_bfloat16 *src0 = C + (size_t)t * kAbTile + c16 * 8;
    for (int k = r; k < Kp; k += 4) {
        const __nv_bfloat16 *src = src0 + (size_t)sJa[k] * lbp;
        const uint32_t dst = dst0 + k * 128 + ((c16 ^ (k & 7)) << 4);
#pragma unroll
        for (int s = 0; s < NP; ++s)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + s * Kp * 128), "l"(src + s * plane) : "memory");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

}  // namespace tbsci
