// Warp-level matrix pieces of the chunkwise backward kernels: mma.sync m16n8k16 (bf16 operands, fp32 accumulation) with every
// derived operand carried as three bf16 values.
//
// Precision.  q, k, v, dO are exact bf16 operands.  A derived fp32 value x is split into h + m + l, each the bf16 rounding of
// what the ones before it leave: 24 significand bits, as many as x has.  A product of an exact with a derived operand is then
// three instructions, one of two derived operands six (the terms below 2^-24 are dropped).
//
// The sums inside an instruction are truncated, not rounded: 1 + 0.75 ulp gives 1, 1 - 0.25 ulp gives 1 - 0.5 ulp, and sixteen
// addends of 2^-26 leave 1 as it is (measured; two bits below the last place of the largest addend are kept).  On random data an
// instruction that adds to a sum of its own size is off by 0.27 ulp towards zero in the mean; errors of one sign add up over a
// long sum.  So the terms of the lower planes have accumulators of their own, and where a result is added to something larger
// or is a long sum itself, the parts are added in fp32.
//
// Why mma.sync and not tcgen05 here: its operands and accumulators live in registers, so a chain of products needs no round
// trip through tensor memory, no shared-memory operand tiles for the derived factor and no barrier between the warps of a
// block; each warp owns 16 columns of the state and runs the whole chunk by itself.  Measured rate on this part: 1 023
// multiply-adds per cycle and SM (8.2 cycles per instruction and scheduler, 20.7 cycles latency), eight times the fp32 pipe.
//
// Tiles in shared memory have rows of 128 bytes (64 bf16) with the 16-byte pieces of a row permuted (sw128), so that the eight
// rows an ldmatrix reads fall into different banks; wider matrices are a sequence of such 64-column blocks.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "common.cuh"

namespace kla {
namespace wmm {

__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

// Fragment loads from a 64-column tile at shared address `t`.
// A operand, 16 x 16 at (m0, k0): tile stored [m][k] (frag_a) or [k][m] (frag_at).
__device__ __forceinline__ void frag_a(uint32_t (&r)[4], uint32_t t, int m0, int k0, int lane)
{
    ldsm4(r, t + sw128(m0 + (lane & 15), (k0 >> 3) + (lane >> 4)));
}
__device__ __forceinline__ void frag_at(uint32_t (&r)[4], uint32_t t, int m0, int k0, int lane)
{
    ldsm4t(r, t + sw128(k0 + (lane & 7) + (lane >> 4) * 8, (m0 >> 3) + ((lane >> 3) & 1)));
}
// B operand, k 16 x n 16 at (k0, n0), registers {b0, b1} of columns n0 .. + 7, then of n0 + 8 .. + 15: tile stored [n][k]
// (frag_b) or [k][n] (frag_bt).
__device__ __forceinline__ void frag_b(uint32_t (&r)[4], uint32_t t, int k0, int n0, int lane)
{
    ldsm4(r, t + sw128(n0 + (lane & 7) + (lane >> 4) * 8, (k0 >> 3) + ((lane >> 3) & 1)));
}
__device__ __forceinline__ void frag_bt(uint32_t (&r)[4], uint32_t t, int k0, int n0, int lane)
{
    ldsm4t(r, t + sw128(k0 + (lane & 15), (n0 >> 3) + (lane >> 4)));
}

// (a, b) as three packed bf16 pairs.
__device__ __forceinline__ void split3(float a, float b, uint32_t &h, uint32_t &m, uint32_t &l)
{
    auto pack = [](float x, float y) {
        const __nv_bfloat162 p = __floats2bfloat162_rn(x, y);
        return *reinterpret_cast<const uint32_t *>(&p);
    };
    h = pack(a, b);
    a -= __uint_as_float(h << 16);
    b -= __uint_as_float(h & 0xffff0000u);
    m = pack(a, b);
    a -= __uint_as_float(m << 16);
    b -= __uint_as_float(m & 0xffff0000u);
    l = pack(a, b);
}
// Two accumulator tiles side by side (16 x 16, columns scaled by the caller) as the three planes of an A operand.
__device__ __forceinline__ void split_a(const float (&x)[4], const float (&y)[4], uint32_t (&h)[4], uint32_t (&m)[4], uint32_t (&l)[4])
{
    split3(x[0], x[1], h[0], m[0], l[0]);
    split3(x[2], x[3], h[1], m[1], l[1]);
    split3(y[0], y[1], h[2], m[2], l[2]);
    split3(y[2], y[3], h[3], m[3], l[3]);
}
// bf16 pair -> two floats
__device__ __forceinline__ float2 unpack(uint32_t x) { return make_float2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)); }

// 16-byte asynchronous copy global -> shared; `in` false writes zeros (nothing is read).
__device__ __forceinline__ void cp16(uint32_t dst, const void *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

}  // namespace wmm
}  // namespace kla
