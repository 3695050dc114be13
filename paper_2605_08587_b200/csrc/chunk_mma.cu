// Chunkwise forward for bf16 inputs (Algorithm 1, right panel; Eqs. 7-9).
//
// One block owns NS = 64 columns of d_v of one (sequence, head) and walks that sequence's chunks (C = 64 tokens) in order.
// Nine warps in three roles, connected by a ring of three chunk slots in shared memory (K, Q, V tiles, operands, per-token scalars):
//
//   chain (4 warps)       the serial dependency over chunks, 16 columns of the state each:
//                             Y_i = R_i - sum_{j<i} X_ij U_j,  R = V - Gam K S            (Eq. 7, by blocks of 16 tokens)
//                             U_i = B_i Y_i + N_ii B_i Y_i
//                             O = Gam Q S + P U                                           (Eq. 8)
//                             S <- gamma_C S + K^T D U,  D = diag(exp(g_C - g_j))         (Eq. 9)
//   prepare (4 warps)     what does not depend on the state, a chunk ahead: decay sums, beta (Eq. 3, ||k||^2 from the diagonal
//                         of K K^T), X = A^- o K K^T, N_ii = (I + B X)_ii^-1 - I, P = A o Q K^T
//   issue (1 warp)        TMA loads and tcgen05 products
//
// Products with the whole state go to tcgen05: [S_hi; S_lo]^T [K; Q]^T, one product of 128 rows (hi and lo parts of 64 columns) and
// 128 columns (the chunk's keys and queries), and [K; Q] K^T.  The serial part runs on mma.sync inside single warps: everything
// transposed, an accumulator tile (16 columns of d_v x tokens or d_k) is at the same time a left operand of the next product, so
// R -> U -> state goes from product to product in registers, without a barrier.  Once per chunk the hi and lo parts of the new state
// go to tensor memory as left operand of the tcgen05 product of the next chunk.
//
// What bounds it: the latency of that chain and the number of instructions in it.  Code that runs once per chunk does not stay in
// the schedulers' instruction caches and issues at about one instruction in three cycles (measured on unrolled against rolled
// copies of the same products).  With all products on mma.sync (504 per chunk and warp at d = 128 instead of 248) a chunk took
// 8 000 cycles; with all of them on tcgen05, whose every product on the chain ends in a hand-over through tensor memory and shared
// memory, 7 400; this way 5 400 (2.73 us, B 8, H 8, d 128, between T 4096 and 8192).  mma.sync stands still while a tcgen05 product
// runs, so the two add up: 400 cycles for [K; Q] K^T, 8 per mma.sync.  [S_hi; S_lo]^T is a left operand in tensor memory: from shared
// memory the state product was bound by the fetch of both operands (8 KB for each 32 cycles of products: 570 cycles), and its
// operand took a proxy fence (headline shape 200.6 -> 194.7 us, 32 packed sequences at d 64 487 -> 472).  The outputs are transposed through
// a buffer that TMA never touches: in the V tile they took such a fence too, in which the warp stood (194.7 -> 188, 472 -> 462).
// The size of the code counts, all the more the more SMs run it: of 70 KB, the two that one short loop to a wait instead of two took out
// were worth 2 % of the headline shape and of 65 536 tokens; two KB more, for tiles of four chunks and two Gram products, gave the
// headline shape 1.6 % (186 -> 183) and cost 65 536 tokens 2.5 % (366 -> 375).
// The outputs on four warps of their own cost more than they took off the chain: 246 us against 201 (82 KB of code instead of 70,
// fetched by all SMs at once, and the Gram product then falls into the block solve).
//
// Precision.  q, k, v are exact bf16 operands.  Every derived operand (S, Y, X, N, P, U) is a pair of bf16 values hi + lo (16
// significand bits; one bf16 rounding of any of them costs 1e-2..7e-2 in max|err|/rms, above the 2e-3 bound), a product of two
// of them hi hi + hi lo + lo hi.  The rounding of a pair is 2.2e-6 of the operand's norm, and so is the term left out.  The block solve
// therefore adds N B Y to B Y in fp32 instead of multiplying Y by (I + N) B: with the identity in the operand U carried three such
// errors of its whole size (2-norm errors of final state and output 5.1e-6 and 6.3e-6; this way 2.5e-6 and 4.5e-6).  In a chunk
// with a near-zero key (beta above HOT_BETA) U has a third part in P U: the rounding of such a token's huge U is the largest error
// of all.  (In every chunk it would cost 8 %.)
//
// mma.sync truncates its sums: used as the accumulator, the state would lose a fraction of a unit in the last place, always towards
// zero, with each of eight products per chunk, which adds up where little is forgotten (log alpha = 0, eta 1e-3, 16 384 tokens: 6e-5
// of the state's norm, now 1.4e-6).  K^T D U is therefore summed by itself, and gamma_C S + that is one fp32 operation per chunk; the
// fp32 state waits in tensor memory meanwhile (registers hold one of the two; 2 % at d = 128, -2 % at d = 64 with two blocks per SM).
//
// Every wait is bounded; when one gives up the block raises an abort flag, reports KLA_ERR_TIMEOUT through the status word,
// lets its copies and products finish and exits.
#include <cuda.h>

#include <cstddef>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "mma_pieces.cuh"
#include "scan_pieces.cuh"
#include "umma.cuh"

namespace kla {

namespace {

using wmm::ldsm4t;
using wmm::unpack;
using namespace umma;

constexpr int C = 64;         // chunk length
constexpr int NS = 64;        // state columns per block
constexpr int CHAIN_T = 128, PREP_T = 128, NT = CHAIN_T + PREP_T + 128;   // (the last warpgroup: one warp works)
constexpr uint32_t WAIT_LIMIT = 2000000000u;   // SM clocks (~1 s) before a wait gives up
constexpr float LOG2E = 1.4426950408889634f;
// The write weights exp(g_C - g_j) are kept above 2^-DEC_FLOOR_LOG2 (~1e-35): U is carried as D U throughout, with D^-1 in X and
// P, and with the floor neither factor leaves the fp32 / bf16 exponent range however strong the decay.  A floored weight puts at
// most 1e-35 of a token into the state instead of less.
constexpr float DEC_FLOOR_LOG2 = 115.f;
constexpr float HOT_BETA = 4096.f;   // q k beta up to ||q|| sqrt(beta) = 64 ||q||: 2^-18 of that is below the other errors
constexpr int LDB = 20;       // row stride (floats) of a 16 x 16 block in the solve scratch
// TMEM columns: [S_hi; S_lo]^T [K; Q]^T (128), [K; Q] K^T (64), the state in fp32 (D / 2), [S_hi; S_lo]^T as left operand (D / 2):
// warp w: lanes 32 w .. the hi, 32 w + 16 .. the lo parts of its columns of d_v, a column for two of d_k.  d 128 uses 320 columns and,
// as they are given in powers of two, holds all 512: no other block with tensor memory runs beside it on an SM (another one of this
// library would not find the shared memory either).
constexpr uint32_t TM_X = 0, TM_G = 128, TM_S = 192;
template <int D>
constexpr uint32_t TM_A = TM_S + D / 2;
template <int D>
constexpr uint32_t TM_COLS = D == 64 ? 256 : 512;

// Lower triangle of 16 x 16 blocks, in fragment order: the four registers of a right operand, 16 bytes per lane.
__device__ __forceinline__ constexpr int blk(int i, int j) { return i * (i + 1) / 2 + j; }
struct TriOperand {
    uint4 hi[10][32], lo[10][32];
};

template <int D>
struct Slot {
    static constexpr int NB = D / 64;
    // per 64 columns: 64 tokens of K, then 64 of Q, rows of 128 bytes, 128-byte swizzle
    alignas(1024) unsigned char kq[NB * 16384];
    alignas(1024) unsigned char v[8192];        // this block's 64 columns
    TriOperand t, p;                            // D N_ii B and below them -X D^-1; P D^-1 (rows over ||q|| with the normalised read-out)
};
struct alignas(16) Scalars {     // of one chunk
    float ngam[C];               // -exp(g_i)
    float gamq[C];               // exp(g_i) (over ||q_i||)
    float bd[C];                 // beta_i exp(g_C - g_i)
    int hot[2];                  // some beta above HOT_BETA among tokens 0 .. 31, 32 .. 63
};

struct alignas(16) PrepScratch {             // of one prepare warp
    float td[2][16 * LDB];       // X_ii, then T_ii, of its two row blocks; the unused upper right 8 x 8 holds an intermediate
    float bet[32];
};

enum Bar {
    B_FULL = 0,      // + slot: tiles landed
    B_READY = 3,     // + slot: operands and scalars written
    B_DONE = 6,      // + slot: every chain warp is through with it
    B_STATE = 9,     // S^T operand of the next chunk written ...
    B_STATE1 = 13,   // ... its second 64 rows of d_k (d = 128)
    B_X = 10,        // [S_hi; S_lo]^T [K; Q]^T complete
    B_G = 11,        // [K; Q] K^T complete
    B_GFREE = 12,    // ... and read
    B_TD = 14,       // diagonal blocks and beta of prepare warp 1 in its scratch
    B_COUNT = 15
};

// BPS, blocks per SM.  One: three chunk slots, registers for the whole chain.  Two (d = 64, more blocks than SMs): two slots and
// half the registers each, so that one block's products fill the other's latencies.
template <int D, int BPS>
struct Smem {
    static constexpr int NSLOT = BPS == 1 ? 3 : 2;
    Slot<D> slot[NSLOT];
    Scalars scal[NSLOT];
    alignas(16) unsigned char outb[4][C * 32];   // a chain warp's 16 columns of the outputs (bf16) on their way out
    PrepScratch prep[2];
    float g2[4][C];              // log2(e) g_i, a copy for each prepare warp
    float qinv[C];
    alignas(8) uint64_t bar[B_COUNT];
    uint32_t tmem;
    volatile int abort_flag;
};

__device__ __forceinline__ uint32_t clock_lo()
{
    uint32_t t;
    asm volatile("mov.u32 %0, %%clock;" : "=r"(t));
    return t;
}
// Every lane polls; the warp leaves together.
__device__ __forceinline__ bool bar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    bool ok = mbar_try_wait(bar, parity);
    if (!ok) {
        const uint32_t t0 = clock_lo();
#pragma unroll 1
        do {
            ok = mbar_try_wait(bar, parity);
        } while (!ok && !*abort_flag && clock_lo() - t0 < WAIT_LIMIT);
        if (!ok) *abort_flag = 1;
    }
    return __all_sync(0xffffffffu, ok);
}

// mma.sync on accumulator tiles kept as pairs: c[0] row lane / 4, c[1] row lane / 4 + 8, columns 2 (lane % 4), + 1.
__device__ __forceinline__ void mma(float2 (&c)[2], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0].x), "+f"(c[0].y), "+f"(c[1].x), "+f"(c[1].y)
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_first(float2 (&c)[2], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)   // c = a b
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
        : "=f"(c[0].x), "=f"(c[0].y), "=f"(c[1].x), "=f"(c[1].y)
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
// x as packed bf16 hi and lo parts.
__device__ __forceinline__ void split(float2 x, uint32_t &hi, uint32_t &lo)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(x.x, x.y);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    const float2 r = fma2(unpack(hi), f2(-1.f), x);   // exact
    const __nv_bfloat162 l = __floats2bfloat162_rn(r.x, r.y);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}
// Register u (0..3) of the left operand made of tiles x, y side by side: x0, x1, y0, y1.
__device__ __forceinline__ void split_left(const float2 (&x)[2], const float2 (&y)[2], int u, uint32_t (&h)[4], uint32_t (&l)[4])
{
    split(u < 2 ? x[u & 1] : y[u & 1], h[u], l[u]);
}
// Tiles x, y as a right operand whose n index is the accumulator's row: x0, y0, x1, y1.
__device__ __forceinline__ void store_right(TriOperand &o, int b, int lane, const float2 (&x)[2], const float2 (&y)[2])
{
    uint4 h, l;
    split(x[0], h.x, l.x);
    split(y[0], h.y, l.y);
    split(x[1], h.z, l.z);
    split(y[1], h.w, l.w);
    o.hi[b][lane] = h;
    o.lo[b][lane] = l;
}
__device__ __forceinline__ float2 load2(const float *p) { return *reinterpret_cast<const float2 *>(p); }

// Four accumulator tiles in sixteen TMEM columns of the warp's lanes, written (there after a wait::st) and read back.
#define R8(c, x, i) c(x[i][0].x), c(x[i][0].y), c(x[i][1].x), c(x[i][1].y), c(x[i + 1][0].x), c(x[i + 1][0].y), c(x[i + 1][1].x), c(x[i + 1][1].y)
__device__ __forceinline__ void tmem_keep(uint32_t addr, const float2 (*x)[2])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"
                 ::R8("f", x, 0), R8("f", x, 2), "r"(addr) : "memory");
}
__device__ __forceinline__ void tmem_kept(uint32_t addr, float2 (&x)[4][2])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
                 "tcgen05.wait::ld.sync.aligned;" : R8("=f", x, 0), R8("=f", x, 2) : "r"(addr) : "memory");
}
#undef R8
// Two left operands side by side (16 rows, 32 of the contraction) in sixteen TMEM columns of sixteen lanes.
__device__ __forceinline__ void tmem_left(uint32_t addr, const uint32_t (&a)[2][4])
{
    asm volatile("tcgen05.st.sync.aligned.16x128b.x4.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};"
                 ::"r"(a[0][0]), "r"(a[0][1]), "r"(a[0][2]), "r"(a[0][3]), "r"(a[1][0]), "r"(a[1][1]), "r"(a[1][2]), "r"(a[1][3]), "r"(addr) : "memory");
}
// 16 TMEM lanes x 16 columns as two accumulator tiles side by side.
__device__ __forceinline__ void tmem_block(uint32_t addr, float2 (&x)[2], float2 (&y)[2])
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(addr) : "memory");
    x[0] = make_float2(__uint_as_float(r[0]), __uint_as_float(r[1]));
    x[1] = make_float2(__uint_as_float(r[2]), __uint_as_float(r[3]));
    y[0] = make_float2(__uint_as_float(r[4]), __uint_as_float(r[5]));
    y[1] = make_float2(__uint_as_float(r[6]), __uint_as_float(r[7]));
}
// 16 lanes (hi parts) and the 16 after them (lo parts) x 64 columns: their sum as eight accumulator tiles.
__device__ __forceinline__ void tmem_sum(uint32_t addr, float2 (&x)[8][2])
{
    uint32_t h[32], l[32];
#define R8(a, i) "=r"(a[i]), "=r"(a[i + 1]), "=r"(a[i + 2]), "=r"(a[i + 3]), "=r"(a[i + 4]), "=r"(a[i + 5]), "=r"(a[i + 6]), "=r"(a[i + 7])
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%64];\n\t"
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, "
        "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%65];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : R8(h, 0), R8(h, 8), R8(h, 16), R8(h, 24), R8(l, 0), R8(l, 8), R8(l, 16), R8(l, 24)
        : "r"(addr), "r"(addr + (16u << 16)) : "memory");
#undef R8
#pragma unroll
    for (int t = 0; t < 8; ++t)
#pragma unroll
        for (int e = 0; e < 2; ++e)
            x[t][e] = add2(make_float2(__uint_as_float(h[4 * t + 2 * e]), __uint_as_float(h[4 * t + 2 * e + 1])),
                           make_float2(__uint_as_float(l[4 * t + 2 * e]), __uint_as_float(l[4 * t + 2 * e + 1])));
}

// Tiles 0, 1 and tiles 2 .. 7 of the same.
__device__ __forceinline__ void tmem_sum_first(uint32_t addr, float2 (&x)[8][2])
{
    uint32_t h[8], l[8];
#define R8(a, i) "=r"(a[i]), "=r"(a[i + 1]), "=r"(a[i + 2]), "=r"(a[i + 3]), "=r"(a[i + 4]), "=r"(a[i + 5]), "=r"(a[i + 6]), "=r"(a[i + 7])
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%16];\n\t"
        "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%8, %9, %10, %11, %12, %13, %14, %15}, [%17];\n\t"
        "tcgen05.wait::ld.sync.aligned;" : R8(h, 0), R8(l, 0) : "r"(addr), "r"(addr + (16u << 16)) : "memory");
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int e = 0; e < 2; ++e)
            x[t][e] = add2(make_float2(__uint_as_float(h[4 * t + 2 * e]), __uint_as_float(h[4 * t + 2 * e + 1])),
                           make_float2(__uint_as_float(l[4 * t + 2 * e]), __uint_as_float(l[4 * t + 2 * e + 1])));
}
__device__ __forceinline__ void tmem_sum_rest(uint32_t addr, float2 (&x)[8][2])
{
    uint32_t h[24], l[24];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%48];\n\t"
        "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%24, %25, %26, %27, %28, %29, %30, %31}, [%49];\n\t"
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23}, [%50];\n\t"
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47}, [%51];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : R8(h, 0), R8(h, 8), R8(h, 16), R8(l, 0), R8(l, 8), R8(l, 16)
        : "r"(addr + 16), "r"(addr + 16 + (16u << 16)), "r"(addr + 32), "r"(addr + 32 + (16u << 16)) : "memory");
#undef R8
#pragma unroll
    for (int t = 0; t < 6; ++t)
#pragma unroll
        for (int e = 0; e < 2; ++e)
            x[t + 2][e] = add2(make_float2(__uint_as_float(h[4 * t + 2 * e]), __uint_as_float(h[4 * t + 2 * e + 1])),
                               make_float2(__uint_as_float(l[4 * t + 2 * e]), __uint_as_float(l[4 * t + 2 * e + 1])));
}

// What a block works on; see ChunkParams for the segment passes.
struct Work {
    int tok0, len;        // first token (of the warm-up run where there is one) and tokens from there
    int first_out;        // leading chunks whose outputs are not stored
    const float *init;    // state before the first token, this head (null: zero); `ident`: the identity
    float *fin;           // where the final state goes, this head (null: nowhere)
    bool ident;
    int h, sl;
};
// Returns false when there is nothing to do (the other kind of pass does the work, or an empty sequence, done here).
template <int D>
__device__ bool find_work(const ChunkParams &params, Work &w)
{
    ChunkParams p = params;
    if (p.seg_pass == 7) {
        if (p.cu_seqlens[p.n_seq + 1] == 1) {
            p.seg_pass = 4;
        } else {
            p.seg_pass = 3;
            p.init_state = p.map_state;
        }
    }
    constexpr int SLICES = D / NS;
    if (p.seg_pass == 6) {
        if (p.seq_order[p.seg_G] != 0) return false;
    } else if (p.seg_pass != 0 && (p.seg_pass >= 4) != (p.cu_seqlens[p.n_seq + 1] == 1)) {
        return false;
    }
    const int nslices = p.seg_pass == 1 ? 2 * SLICES : SLICES;
    const int sl2 = blockIdx.x % nslices;
    w.ident = sl2 >= SLICES;
    w.sl = sl2 % SLICES;
    w.h = (blockIdx.x / nslices) % p.H;
    int n = blockIdx.x / (nslices * p.H);
    if (p.seg_pass == 1) n = (n / (p.seg_G - 1)) * p.seg_G + n % (p.seg_G - 1);
    else if ((p.seg_pass == 0 || p.seg_pass == 6) && p.seq_order) n = p.seq_order[n];   // packed input: longest sequences first
    if (p.cu_seqlens) {
        w.tok0 = p.cu_seqlens[n];
        w.len = p.cu_seqlens[n + 1] - w.tok0;
    } else {
        w.tok0 = n * p.T;
        w.len = p.T;
    }
    auto state = [&](int sq) { return ((size_t)sq * p.H + w.h) * D * D; };
    const int32_t *warm = p.cu_seqlens + p.n_seq + 2;   // warm-up lengths (passes 4 and 5), then the piece table (pass 5)
    bool early = false;
    int sq = n;                                          // index of the states this block reads ...
    if (p.seg_pass == 5) {
        const int32_t piece = warm[p.n_seq * p.H + n];
        sq = piece & 0x1fffffff;
        early = !((piece >> 29) & 1);                    // not a sequence's first piece
        w.fin = p.final_state && ((piece >> 30) & 1) ? p.final_state + state(sq) : nullptr;
    } else if (p.seg_pass == 3 || p.seg_pass == 4) {
        if (p.seg_pass == 4) {
            sq = n / p.seg_G;
            early = n % p.seg_G != 0;
        }
        w.fin = p.final_state && n % p.seg_G == p.seg_G - 1 ? p.final_state + state(n / p.seg_G) : nullptr;
    } else {
        float *f = w.ident ? p.map_state : p.final_state;
        w.fin = f ? f + state(n) : nullptr;
    }
    w.init = p.init_state && !early && p.seg_pass != 1 ? p.init_state + state(sq) : nullptr;
    w.first_out = 0;
    if (early) {   // from zero, so many chunks before the piece
        w.first_out = warm[n * p.H + w.h];
        w.tok0 -= w.first_out * C;
        w.len += w.first_out * C;
    }
    if (w.len > 0) return true;
    if (p.final_state) {   // empty sequence: the final state is the initial state (never a segment: those are not empty)
        const size_t off = state(n) + (size_t)w.sl * NS;
        for (int i = threadIdx.x; i < D * (NS / 4); i += NT) {
            const size_t e = off + (size_t)(i / (NS / 4)) * D + (i % (NS / 4)) * 4;
            store4(p.final_state + e, p.init_state ? load4(p.init_state + e) : make_float4(0.f, 0.f, 0.f, 0.f));
        }
    }
    return false;
}

// ---- prepare --------------------------------------------------------------------------------------------------------------
// [K; Q] K^T lies in TMEM with its rows as lanes, 32 per warp: warps 0 and 1 form X (token blocks 0, 1 and 2, 3) and the diagonal
// blocks N, warps 2 and 3 P.  Blocks of 16 x 16 are read, weighted and stored as operands one after the other in a rolled
// loop.  (I + B X)_ii^-1 by 8 x 8 substitution (a column per lane) and one merge; the rest of the triangular solve is
// left to the chain, which takes U block by block: as many products there as with the whole inverse, and the block products of
// the inverse, longer than everything else here, are not needed.  Warp 1 has the most blocks and the chain waits for it, so warp 2,
// which has the fewest, inverts its diagonal blocks for it (32 packed sequences, d 64, two blocks per SM: -3 %).
template <int D, int BPS, bool VAR>
__device__ void prepare(const ChunkParams &p, Smem<D, BPS> &sm, const Work &wk, int nchunks)
{
    constexpr int NB = D / 64, NSLOT = Smem<D, BPS>::NSLOT;
    const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & 3;
    const int g = lane >> 2, t2 = 2 * (lane & 3);
    const int h = wk.h;
    const bool isx = w < 2;
    const uint32_t tg = sm.tmem + TM_G + ((uint32_t)(32 * w) << 16);
    PrepScratch &sc = sm.prep[w & 1];
    float *g2 = sm.g2[w];

    // log alpha of tokens 2 lane, 2 lane + 1; eta of the warp's token blocks (X warps), tokens g, g + 8 of each: a chunk ahead
    float la[2], et[4];
    auto fetch = [&](int c) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = c * C + 2 * lane + u;
            la[u] = i < wk.len ? p.log_alpha[(size_t)(wk.tok0 + i) * p.H + h] : 0.f;
        }
        if (isx) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e = c * C + 32 * w + g + 8 * u;
                et[u] = e < wk.len ? p.eta[(size_t)(wk.tok0 + e) * p.H + h] : 0.f;
            }
        }
    };
    fetch(0);

    for (int c = 0; c < nchunks; ++c) {
        const int s = c % NSLOT;
        Slot<D> &sl = sm.slot[s];
        const int rows = min(C, wk.len - c * C);
        // decay sums (every warp finds the same values; lane l holds tokens 2l, 2l + 1)
        float incl = la[0] + la[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const float gc2 = __shfl_sync(0xffffffffu, incl, 31) * LOG2E, ga2 = (incl - la[1]) * LOG2E, gb2 = incl * LOG2E;
        const float e4[4] = {et[0], et[1], et[2], et[3]};
        *reinterpret_cast<float2 *>(&g2[2 * lane]) = make_float2(ga2, gb2);
        if (c + 1 < nchunks) fetch(c + 1);
        auto floored = [&](float2 x) { return make_float2(fmaxf(gc2, x.x - DEC_FLOOR_LOG2), fmaxf(gc2, x.y - DEC_FLOOR_LOG2)); };
        const bool qnorm = VAR && (p.variant & VARIANT_QNORM);
        // the product is there: so are the tiles, and the slot's last user is through
        if (!bar_wait(&sm.bar[B_G], c & 1, &sm.abort_flag)) break;
        tc_fence_after();
        if (!isx) {
            if (qnorm) {   // a token per lane
                float n = 0.f;
                const int r = 32 * (w - 2) + lane;
#pragma unroll 1
                for (int e = 0; e < NB * 8; ++e) {
                    const uint4 raw = *reinterpret_cast<const uint4 *>(sl.kq + (e >> 3) * 16384 + 8192 + sw128(r, e & 7));
                    const uint32_t x[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float2 f = unpack(x[u]);
                        n += f.x * f.x + f.y * f.y;
                    }
                }
                sm.qinv[r] = 1.f / sqrtf(n);
                __syncwarp();
            }
            if ((lane >> 4) == w - 2) {   // per-token scalars
                float2 gm = make_float2(ex2_approx(ga2), ex2_approx(gb2));
                *reinterpret_cast<float2 *>(&sm.scal[s].ngam[2 * lane]) = make_float2(-gm.x, -gm.y);
                if (qnorm) gm = mul2(gm, load2(&sm.qinv[2 * lane]));
                *reinterpret_cast<float2 *>(&sm.scal[s].gamq[2 * lane]) = gm;
            }
        }
        __syncwarp();

        float2 x[2], y[2];
        if (isx) {
            // the two diagonal blocks: ||k||^2 and X_ii
#pragma unroll 1
            for (int rb = 0; rb < 2; ++rb) {
                const int i0 = 32 * w + 16 * rb;
                tmem_block(tg + ((uint32_t)(16 * rb) << 16) + i0, x, y);
                // token g: tile x, row half 0; token g + 8: tile y, row half 1; at the lane whose columns are g & ~1, g | 1
                if ((lane & 3) == (g >> 1)) {
                    const float n0 = ((g & 1) ? x[0].y : x[0].x) + p.eps, n1 = ((g & 1) ? y[1].y : y[1].x) + p.eps;
                    const float a0 = rb ? e4[2] : e4[0], a1 = rb ? e4[3] : e4[1];
                    const bool plain = VAR && (p.variant & VARIANT_COEFF_ETA);
                    sc.bet[16 * rb + g] = i0 + g < rows ? (plain ? a0 : a0 / n0) : 0.f;
                    sc.bet[16 * rb + g + 8] = i0 + g + 8 < rows ? (plain ? a1 : a1 / n1) : 0.f;
                }
                const float r0 = g2[i0 + g], r1 = g2[i0 + g + 8];
                const float2 c0 = load2(&g2[i0 + t2]), c1 = load2(&g2[i0 + 8 + t2]);
                const bool v0 = i0 + g < rows, v1 = i0 + g + 8 < rows;
                float *td = sc.td[rb] + g * LDB + t2;
                *reinterpret_cast<float2 *>(td) = make_float2(v0 && t2 < g ? ex2_approx(r0 - c0.x) * x[0].x : 0.f, v0 && t2 + 1 < g ? ex2_approx(r0 - c0.y) * x[0].y : 0.f);
                *reinterpret_cast<float2 *>(td + 8 * LDB) = make_float2(v1 ? ex2_approx(r1 - c0.x) * x[1].x : 0.f, v1 ? ex2_approx(r1 - c0.y) * x[1].y : 0.f);
                *reinterpret_cast<float2 *>(td + 8 * LDB + 8) = make_float2(v1 && t2 < g ? ex2_approx(r1 - c1.x) * y[1].x : 0.f, v1 && t2 + 1 < g ? ex2_approx(r1 - c1.y) * y[1].y : 0.f);
            }
            __syncwarp();
            {
                const bool hot = __any_sync(0xffffffffu, sc.bet[lane] > HOT_BETA);
                if (lane == 0) sm.scal[s].hot[w] = hot;
            }
            __syncwarp();
            if (w == 1 && lane == 0) mbar_arrive(&sm.bar[B_TD]);
        }
        // -X D^-1 below the diagonal blocks, P D^-1 up to them
        const bool qn = qnorm && !isx;
#pragma unroll 1
        for (int rb = 0; rb < 2; ++rb) {
            const int bi = 2 * (w & 1) + rb, i0 = 16 * bi;
            const float r0 = g2[i0 + g], r1 = g2[i0 + g + 8];
            const float f0 = isx ? -1.f : qn ? sm.qinv[i0 + g] : 1.f, f1 = isx ? -1.f : qn ? sm.qinv[i0 + g + 8] : 1.f;
            const bool v0 = !isx || i0 + g < rows, v1 = !isx || i0 + g + 8 < rows;   // (a row past the end may hold anything)
            const int nb = isx ? bi : bi + 1;
#pragma unroll 1
            for (int j = 0; j < nb; ++j) {
                tmem_block(tg + ((uint32_t)(16 * rb) << 16) + 16 * j, x, y);
                const float2 c0 = floored(load2(&g2[16 * j + t2])), c1 = floored(load2(&g2[16 * j + 8 + t2]));
                const int lim = j == bi ? g : 16;   // columns up to the row on the diagonal block
                x[0].x = v0 && t2 <= lim ? f0 * ex2_approx(r0 - c0.x) * x[0].x : 0.f;
                x[0].y = v0 && t2 < lim ? f0 * ex2_approx(r0 - c0.y) * x[0].y : 0.f;
                x[1].x = v1 ? f1 * ex2_approx(r1 - c0.x) * x[1].x : 0.f;
                x[1].y = v1 ? f1 * ex2_approx(r1 - c0.y) * x[1].y : 0.f;
                y[0].x = v0 && lim == 16 ? f0 * ex2_approx(r0 - c1.x) * y[0].x : 0.f;
                y[0].y = v0 && lim == 16 ? f0 * ex2_approx(r0 - c1.y) * y[0].y : 0.f;
                y[1].x = v1 && t2 <= lim ? f1 * ex2_approx(r1 - c1.x) * y[1].x : 0.f;
                y[1].y = v1 && t2 < lim ? f1 * ex2_approx(r1 - c1.y) * y[1].y : 0.f;
                store_right(isx ? sl.t : sl.p, blk(bi, j), lane, x, y);
            }
        }
        // the inverses of the diagonal blocks: warp 0 those of its own, warp 2, which has the fewest blocks, those of warp 1
        if (!(w & 1)) {
            if (w == 2 && !bar_wait(&sm.bar[B_TD], c & 1, &sm.abort_flag)) break;
            PrepScratch &si = sm.prep[w >> 1];
            // 8 x 8 diagonal blocks by substitution: lane l solves column l % 8 of block l / 8 of four
            float xs[8];
            {
                const int b8 = lane >> 3, col = lane & 7;
                float *td = si.td[b8 >> 1] + (b8 & 1) * (8 * LDB + 8);
                const float4 bl = load4(si.bet + b8 * 8), bh = load4(si.bet + b8 * 8 + 4);
                const float bb[8] = {bl.x, bl.y, bl.z, bl.w, bh.x, bh.y, bh.z, bh.w};
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    float a = 0.f;
                    if (r > 0) {
                        const float4 f0 = load4(td + r * LDB), f1 = r > 4 ? load4(td + r * LDB + 4) : make_float4(0.f, 0.f, 0.f, 0.f);
                        const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
#pragma unroll
                        for (int m = 0; m < r; ++m) a += f[m] * xs[m];
                    }
                    xs[r] = r == col ? 1.f : (r > col ? -bb[r] * a : 0.f);
                }
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 8; ++r) td[r * LDB + col] = xs[r];
            }
            __syncwarp();
            // T_10 = -T_11 (B_1 X_10 T_00): row g, columns t2, t2 + 1 of both blocks
#pragma unroll 1
            for (int rb = 0; rb < 2; ++rb) {
                const float *td = si.td[rb];
                const float4 f0 = load4(td + (8 + g) * LDB), f1 = load4(td + (8 + g) * LDB + 4);
                const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
                float2 a = f2(0.f);
#pragma unroll
                for (int m = 0; m < 8; ++m) a = fma2(f2(f[m]), load2(td + m * LDB + t2), a);
                *reinterpret_cast<float2 *>(si.td[rb] + g * LDB + 8 + t2) = mul2(f2(-si.bet[16 * rb + 8 + g]), a);
            }
            __syncwarp();
#pragma unroll 1
            for (int rb = 0; rb < 2; ++rb) {
                const float *td = si.td[rb];
                const float4 f0 = load4(td + (8 + g) * LDB + 8), f1 = load4(td + (8 + g) * LDB + 12);
                const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
                float2 a = f2(0.f);
#pragma unroll
                for (int m = 0; m < 8; ++m) a = fma2(f2(f[m]), load2(td + m * LDB + 8 + t2), a);
                const float2 c0 = load2(&si.bet[16 * rb + t2]), c1 = load2(&si.bet[16 * rb + 8 + t2]);
                const int i0 = 16 * (w + rb) + g;
                const float2 d0 = f2(ex2_approx(fmaxf(gc2 - g2[i0], -DEC_FLOOR_LOG2))), d1 = f2(ex2_approx(fmaxf(gc2 - g2[i0 + 8], -DEC_FLOOR_LOG2)));
                x[0] = mul2(mul2(load2(td + g * LDB + t2), c0), d0);
                x[1] = mul2(mul2(a, c0), d1);
                y[0] = f2(0.f);
                y[1] = mul2(mul2(load2(td + (8 + g) * LDB + 8 + t2), c1), d1);
                // the diagonal, D B, stays in fp32
                const bool e0 = t2 == g, e1 = t2 + 1 == g;
                if (e0 || e1) {
                    sm.scal[s].bd[i0] = e0 ? x[0].x : x[0].y;
                    sm.scal[s].bd[i0 + 8] = e0 ? y[1].x : y[1].y;
                }
                x[0] = make_float2(e0 ? 0.f : x[0].x, e1 ? 0.f : x[0].y);
                y[1] = make_float2(e0 ? 0.f : y[1].x, e1 ? 0.f : y[1].y);
                store_right(sl.t, blk(w + rb, w + rb), lane, x, y);
            }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.bar[B_GFREE]);   // (of warp 2 also: the scratch of warp 1 has been read)
        if (rows < C) {   // K rows past the end of the sequence hold a neighbour's tokens: inert from here on
            for (int e = threadIdx.x & 127; e < (C - rows) * 8; e += PREP_T) {
                const uint32_t off = sw128(rows + (e >> 3), e & 7);
#pragma unroll
                for (int kb = 0; kb < NB; ++kb) *reinterpret_cast<uint4 *>(sl.kq + kb * 16384 + off) = make_uint4(0, 0, 0, 0);
            }
        }
        __syncwarp();
        bool signal = true;
        if (VAR) signal = !(p.variant & VARIANT_TEST_TIMEOUT);   // test hook: the chain's bounded wait then runs out
        if (lane == 0 && signal) mbar_arrive(&sm.bar[B_READY + s]);
    }
}

// ---- chain ----------------------------------------------------------------------------------------------------------------
// OUT = void: no outputs (segment pass 1).  A warp has its scheduler almost to itself and issues in order, so what waits for
// nothing is placed between what does: the state update and the outputs of token block j - 1 cover the solve of block j, and the
// outputs leave while the next chunk's state product runs.
template <int D, int BPS, typename OUT>
__device__ void chain(const ChunkParams &p, Smem<D, BPS> &sm, const Work &wk, int nchunks)
{
    constexpr bool HAS_OUT = !std::is_void<OUT>::value;
    using Elem = typename std::conditional<HAS_OUT, OUT, char>::type;
    constexpr int KS = D / 16, NSLOT = Smem<D, BPS>::NSLOT;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int g = lane >> 2, t2 = 2 * (lane & 3);
    const int dv = wk.sl * NS + 16 * w + g;   // columns dv, dv + 8 of d_v
    // S[t][e]: rows 8 t + t2, + 1 of d_k, column dv + 8 e: the state, during a chunk K^T D U of the tokens so far
    float2 S[D / 8][2];
#pragma unroll
    for (int t = 0; t < D / 8; ++t)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int r = 8 * t + t2, cc = dv + 8 * e;
            S[t][e] = wk.init ? make_float2(wk.init[(size_t)r * D + cc], wk.init[(size_t)(r + 1) * D + cc])
                              : make_float2(wk.ident && r == cc ? 1.f : 0.f, wk.ident && r + 1 == cc ? 1.f : 0.f);
        }
    const uint32_t tx = sm.tmem + TM_X + ((uint32_t)(32 * w) << 16);
    // per-lane parts of the tile addresses: right operands K (16 tokens x 16 of d_k); V
    uint32_t ktx[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) ktx[u] = sw128(lane & 15, 2 * u + (lane >> 4));
    const uint32_t ob = smem_u32(sm.outb[w]) + ((lane & 7) + (lane >> 4) * 8) * 32 + ((((lane >> 3) & 1) ^ ((lane >> 2) & 1)) << 4);
    const uint32_t vtx = sw128((lane & 7) + (lane >> 4) * 8, 2 * w + ((lane >> 3) & 1));

    const uint32_t ta = sm.tmem + TM_A<D> + ((uint32_t)(32 * w) << 16);
    auto store_state = [&](int q) {   // rows 32 q .. of d_k
        uint32_t h[2][4], l[2][4];
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
            for (int u = 0; u < 4; ++u) split_left(S[4 * q + 2 * v], S[4 * q + 2 * v + 1], u, h[v], l[v]);
        tmem_left(ta + 16 * q, h);
        tmem_left(ta + 16 * q + (16u << 16), l);
    };
    // d = 128: the product over the first 64 rows of d_k starts while the others are being finished (-1.5 %)
    auto state_written = [&](int part) {
        tmem_wait_stores();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.bar[part ? B_STATE1 : B_STATE]);
    };
#pragma unroll
    for (int q = 0; q < KS / 2; ++q) store_state(q);
    const uint32_t ts = sm.tmem + TM_S + ((uint32_t)(32 * w) << 16);
#pragma unroll
    for (int ks = 0; ks < KS; ks += 2) tmem_keep(ts + 8 * ks, &S[2 * ks]);
    if (D == 128) state_written(1);
    state_written(0);

    const size_t tok_stride = (size_t)p.H * D;
    Elem *out = static_cast<Elem *>(p.out) + ((size_t)wk.tok0 * p.H + wk.h) * D + wk.sl * NS + 16 * w;
    for (int c = 0; c < nchunks; ++c) {
        const int s = c % NSLOT;
        Slot<D> &sl = sm.slot[s];
        const int rows = min(C, wk.len - c * C);
        if (!bar_wait(&sm.bar[B_READY + s], (c / NSLOT) & 1, &sm.abort_flag)) break;
        const uint32_t kt = smem_u32(sl.kq), vt = smem_u32(sl.v) + vtx;
        uint32_t vv[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (!wk.ident) ldsm4t(vv[j], vt + j * 2048);
            else vv[j][0] = vv[j][1] = vv[j][2] = vv[j][3] = 0;
        }
        if (!bar_wait(&sm.bar[B_X], c & 1, &sm.abort_flag)) break;
        tc_fence_after();

        float2 x[8][2];   // K S, then R, then Y, then D U
        tmem_sum_first(tx, x);
        auto residual = [&](int t) {   // R = V - Gam K S, 8 tokens
            const float2 gm = load2(&sm.scal[s].ngam[8 * t + t2]);
            x[t][0] = fma2(gm, x[t][0], unpack(vv[t >> 1][2 * (t & 1)]));
            x[t][1] = fma2(gm, x[t][1], unpack(vv[t >> 1][2 * (t & 1) + 1]));
        };
        auto live_only = [&](int t) {   // nothing from tokens past the end
            if (8 * t + t2 >= rows) x[t][0].x = x[t][1].x = 0.f;
            if (8 * t + t2 + 1 >= rows) x[t][0].y = x[t][1].y = 0.f;
        };
        float2 o[8][2];   // Gam Q S, then O
        uint32_t rh[4], rl[4], uh[2][4], ul[2][4];   // operands Y_j, D U_j
        const bool hot = HAS_OUT && (sm.scal[s].hot[0] | sm.scal[s].hot[1]);
        uint32_t b[2][2][4];
        auto fetch_k = [&](int q) {   // K as right operand: step q = (16 tokens, 32 of d_k)
            const int j = q / (KS / 2), n = 2 * (q % (KS / 2));
#pragma unroll
            for (int u = 0; u < 2; ++u) ldsm4t(b[q & 1][u], kt + ktx[(n + u) & 3] + ((n + u) >> 2) * 16384 + j * 2048);
        };
        // += (D U_j)^T K_j, 32 rows of d_k; `extra` between the products
        auto update = [&](int q, auto &&extra) {
            const int j = q / (KS / 2), n = 2 * (q % (KS / 2));
            if (q + 1 < 2 * KS) fetch_k(q + 1);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                if (j == 0) {
                    mma_first(S[2 * (n + u)], uh[0], b[q & 1][u][0], b[q & 1][u][1]);
                    mma_first(S[2 * (n + u) + 1], uh[0], b[q & 1][u][2], b[q & 1][u][3]);
                } else {
                    mma(S[2 * (n + u)], uh[j & 1], b[q & 1][u][0], b[q & 1][u][1]);
                    mma(S[2 * (n + u) + 1], uh[j & 1], b[q & 1][u][2], b[q & 1][u][3]);
                }
            }
            extra();
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                mma(S[2 * (n + u)], ul[j & 1], b[q & 1][u][0], b[q & 1][u][1]);
                mma(S[2 * (n + u) + 1], ul[j & 1], b[q & 1][u][2], b[q & 1][u][3]);
            }
        };
        auto outputs = [&](int j) {   // O += (P_.j D^-1) (D U_j)
            if constexpr (HAS_OUT) {
                uint4 f[4];
#pragma unroll
                for (int i = j; i < 4; ++i) f[i] = sl.p.hi[blk(i, j)][lane];
#pragma unroll
                for (int tm = 0; tm < 3; ++tm)
#pragma unroll
                    for (int i = j; i < 4; ++i) {
                        mma(o[2 * i], tm == 1 ? ul[j & 1] : uh[j & 1], f[i].x, f[i].y);
                        mma(o[2 * i + 1], tm == 1 ? ul[j & 1] : uh[j & 1], f[i].z, f[i].w);
                        if (tm == 1) f[i] = sl.p.lo[blk(i, j)][lane];
                    }
                if (hot) {   // what hi and lo leave of U_j
                    uint32_t m[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float2 r = fma2(unpack(ul[j & 1][u]), f2(-1.f), fma2(unpack(uh[j & 1][u]), f2(-1.f), x[2 * j + (u >> 1)][u & 1]));
                        const __nv_bfloat162 mm = __floats2bfloat162_rn(r.x, r.y);
                        m[u] = *reinterpret_cast<const uint32_t *>(&mm);
                    }
#pragma unroll
                    for (int i = j; i < 4; ++i) {
                        const uint4 ph = sl.p.hi[blk(i, j)][lane];
                        mma(o[2 * i], m, ph.x, ph.y);
                        mma(o[2 * i + 1], m, ph.z, ph.w);
                    }
                }
            }
        };
        constexpr int QJ = KS / 2, QH = QJ / 2;   // update steps per token block, and half of them
        residual(0);
        residual(1);
        if (rows < C) {
            live_only(0);
            live_only(1);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) split_left(x[0], x[1], u, rh, rl);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            // D U_j = D B Y_j + (D N_jj B) Y_j
            {
                const uint4 th = sl.t.hi[blk(j, j)][lane], tl = sl.t.lo[blk(j, j)][lane];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float2 bd = load2(&sm.scal[s].bd[16 * j + 8 * u + t2]);
                    x[2 * j + u][0] = mul2(bd, x[2 * j + u][0]);
                    x[2 * j + u][1] = mul2(bd, x[2 * j + u][1]);
                }
                mma(x[2 * j], rh, th.x, th.y);
                mma(x[2 * j + 1], rh, th.z, th.w);
                mma(x[2 * j], rl, th.x, th.y);
                mma(x[2 * j + 1], rl, th.z, th.w);
                mma(x[2 * j], rh, tl.x, tl.y);
                mma(x[2 * j + 1], rh, tl.z, tl.w);
            }
            if (j == 0) {
                tmem_sum_rest(tx, x);
#pragma unroll
                for (int t = 2; t < 8; ++t) residual(t);
                if (rows < C) {
#pragma unroll
                    for (int t = 2; t < 8; ++t) live_only(t);
                }
            } else {
#pragma unroll
                for (int q = 0; q < QH; ++q) update((j - 1) * QJ + q, [] {});
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) split_left(x[2 * j], x[2 * j + 1], u, uh[j & 1], ul[j & 1]);
            // Y_i -= (X_ij D^-1) (D U_j)
            if (j < 3) {
                uint4 f[3];
#pragma unroll
                for (int i = j + 1; i < 4; ++i) f[i - j - 1] = sl.t.hi[blk(i, j)][lane];
#pragma unroll
                for (int tm = 0; tm < 3; ++tm) {
                    if (tm == 2) {
#pragma unroll
                        for (int i = j + 1; i < 4; ++i) f[i - j - 1] = sl.t.lo[blk(i, j)][lane];
                    }
#pragma unroll
                    for (int i = j + 1; i < 4; ++i) {
                        const uint4 &ff = f[i - j - 1];
                        mma(x[2 * i], tm == 1 ? ul[j & 1] : uh[j & 1], ff.x, ff.y);
                        mma(x[2 * i + 1], tm == 1 ? ul[j & 1] : uh[j & 1], ff.z, ff.w);
                    }
                }
            }
            if (j == 0) {
                fetch_k(0);
                if (HAS_OUT) {
                    tmem_sum(tx + 64, o);
#pragma unroll
                    for (int t = 0; t < 8; ++t) {
                        const float2 gq = load2(&sm.scal[s].gamq[8 * t + t2]);
                        o[t][0] = mul2(o[t][0], gq);
                        o[t][1] = mul2(o[t][1], gq);
                    }
                }
            } else {
#pragma unroll
                for (int q = QH; q < QJ; ++q) update((j - 1) * QJ + q, [] {});
                outputs(j - 1);
            }
            if (j < 3) {
#pragma unroll
                for (int u = 0; u < 4; ++u) split_left(x[2 * j + 2], x[2 * j + 3], u, rh, rl);
            }
        }
        outputs(3);
        // the last token block, and the finished rows of the state, gC S + K^T D U, on their way to the next product
        const float2 gC = f2(-sm.scal[s].ngam[C - 1]);
        auto finish = [&](int q) {   // 32 rows
            float2 kept[4][2];
            tmem_kept(ts + 16 * q, kept);
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
                for (int e = 0; e < 2; ++e) S[4 * q + t][e] = fma2(gC, kept[t][e], S[4 * q + t][e]);
            tmem_keep(ts + 16 * q, &S[4 * q]);
            store_state(q);
        };
#pragma unroll
        for (int q = 0; q < QJ; ++q)
            update(3 * QJ + q, [&] {
                if (q > 0) finish(q - 1);
                if (D == 128 && q == QJ / 2 && c + 1 < nchunks) state_written(0);
            });
        finish(QJ - 1);
        if (c + 1 < nchunks) state_written(D == 128);
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.bar[B_DONE + s]);
        if constexpr (HAS_OUT) {
            const int live = c >= wk.first_out ? rows : 0;
            if constexpr (std::is_same<OUT, float>::value) {
#pragma unroll
                for (int t = 0; t < 8; ++t)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        Elem *d = out + (8 * t + t2) * tok_stride + g + 8 * e;
                        if (8 * t + t2 < live) d[0] = o[t][e].x;
                        if (8 * t + t2 + 1 < live) d[tok_stride] = o[t][e].y;
                    }
            } else {
                // transposed through shared memory, so that a store is 16 bytes of one token (a buffer of its own: in a tile that
                // TMA refills it takes a proxy fence, on which the warp then stands)
#pragma unroll
                for (int t = 0; t < 8; t += 2) {
                    uint32_t r[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const __nv_bfloat162 hh = __floats2bfloat162_rn(o[t + (u >> 1)][u & 1].x, o[t + (u >> 1)][u & 1].y);
                        r[u] = *reinterpret_cast<const uint32_t *>(&hh);
                    }
                    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};"
                                 ::"r"(ob + t * 256), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
                }
                __syncwarp();
                const int r0 = lane >> 1, ch = lane & 1;
                const unsigned char *src = sm.outb[w] + r0 * 32 + ((ch ^ ((r0 >> 2) & 1)) << 4);
                Elem *d = out + r0 * tok_stride + ch * 8;
                uint4 r[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) r[e] = *reinterpret_cast<const uint4 *>(src + e * 512);
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (16 * e + r0 < live) *reinterpret_cast<uint4 *>(d + 16 * e * tok_stride) = r[e];
            }
            out += C * tok_stride;
        }
    }
    // The last chunk stores its state to tensor memory like any other, and nobody waits for it: the columns are given back next.
    // (Left out in the last chunk instead, the stores stand behind a branch in every one: headline shape 184.7 -> 190.8 us, 65 536 tokens
    // 362.6 -> 379.9.)
    tmem_wait_stores();
    if (wk.fin && !sm.abort_flag) {
#pragma unroll
        for (int t = 0; t < D / 8; ++t)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float *d = wk.fin + (size_t)(8 * t + t2) * D + dv + 8 * e;
                d[0] = S[t][e].x;
                d[D] = S[t][e].y;
            }
    }
}

// ---- issue ----------------------------------------------------------------------------------------------------------------
// One warp in lock step.  In the order the events fall: the state product of chunk c, [K; Q] K^T of chunk c + 1, the loads of c + 2
// (with two slots those of c + 1, before its [K; Q] K^T).
template <int D, int BPS, bool HAS_OUT>
__device__ void issue(const CUtensorMap *tm_q, const CUtensorMap *tm_k, const CUtensorMap *tm_v, Smem<D, BPS> &sm, const Work &wk, int nchunks)
{
    constexpr int NB = D / 64, NSLOT = Smem<D, BPS>::NSLOT;
    const bool first = (threadIdx.x & 31) == 0;
    auto load = [&](int c) {
        if (first) {
            Slot<D> &sl = sm.slot[c % NSLOT];
            uint64_t *bar = &sm.bar[B_FULL + c % NSLOT];
            mbar_expect_tx(bar, (2 * NB + 1) * 8192);
            const int y = wk.tok0 + c * C;
#pragma unroll
            for (int kb = 0; kb < NB; ++kb) {
                tma_load_2d(sl.kq + kb * 16384, tm_k, wk.h * D + kb * 64, y, bar);
                tma_load_2d(sl.kq + kb * 16384 + 8192, tm_q, wk.h * D + kb * 64, y, bar);
            }
            tma_load_2d(sl.v, tm_v, wk.h * D + wk.sl * NS, y, bar);
        }
        __syncwarp();
    };
    auto wait = [&](int b, int parity) {
        const bool ok = bar_wait(&sm.bar[b], parity & 1, &sm.abort_flag);
        tc_fence_after();
        return ok;
    };
    auto gram = [&](int c) {
        const uint32_t a = desc_lo(smem_desc_sw128(smem_u32(sm.slot[c % NSLOT].kq), 0, 1024));
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) mma4_bf16_lo<2, 2>(sm.tmem + TM_G, a + kb * 1024, a + kb * 1024, idesc_bf16(128, 64, 0, 0), kb > 0);
        mma_commit(&sm.bar[B_G]);
    };
    for (int c = 0; c < NSLOT && c < nchunks; ++c) load(c);
    if (!wait(B_FULL, 0)) return;
    gram(0);
    for (int c = 0; c < nchunks; ++c) {
        if (!wait(B_STATE, c)) return;
        const uint32_t b = desc_lo(smem_desc_sw128(smem_u32(sm.slot[c % NSLOT].kq), 0, 1024));
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) {
            if (kb == 1 && !wait(B_STATE1, c)) return;
            mma4_bf16_ta<2>(sm.tmem + TM_X, sm.tmem + TM_A<D> + kb * 32, b + kb * 1024, idesc_bf16(128, HAS_OUT ? 128 : 64, 0, 0), kb > 0);
        }
        mma_commit(&sm.bar[B_X]);
        auto next_gram = [&]() {
            if (c + 1 >= nchunks) return true;
            if (!wait(B_FULL + (c + 1) % NSLOT, (c + 1) / NSLOT) || !wait(B_GFREE, c)) return false;
            gram(c + 1);
            return true;
        };
        auto next_load = [&]() {   // into the slot of chunk c - 1
            if (c == 0 || c - 1 + NSLOT >= nchunks) return true;
            if (!wait(B_DONE + (c - 1) % NSLOT, (c - 1) / NSLOT)) return false;
            load(c - 1 + NSLOT);
            return true;
        };
        if (NSLOT == 3 ? !next_gram() || !next_load() : !next_load() || !next_gram()) return;
    }
}

// VAR: compiled with the layer-edge variants (beta = eta, read-out over ||q||) and the test hook; the default instantiation
// carries none of their code.
template <int D, int BPS, typename OUT, bool VAR>
__global__ void __launch_bounds__(NT, BPS)
kla_chunk_mma_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                     const __grid_constant__ CUtensorMap tm_v, ChunkParams p)
{
    // Used as declared, not rounded up at run time: the compiler then knows that it is shared memory (rounded up, every access is
    // a generic one: 12 % slower).  There is no static shared memory, so it starts on such a boundary; checked all the same.
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    constexpr int NSLOT = Smem<D, BPS>::NSLOT;
    Smem<D, BPS> &sm = *reinterpret_cast<Smem<D, BPS> *>(smem_dyn);
    static_assert(sizeof(Smem<D, BPS>) <= (BPS == 1 ? 232448 : 115712), "shared memory of one block");
    if (smem_u32(smem_dyn) & 1023) {
        if (threadIdx.x == 0 && p.status_word) atomicExch(p.status_word, (int)KLA_ERR_ALIGN);
        return;
    }
    Work wk;
    if (!find_work<D>(p, wk)) return;
    const int nchunks = (wk.len + C - 1) / C;
    const int tid = threadIdx.x;
    if (tid == 0) {
        for (int s = 0; s < NSLOT; ++s) {
            mbar_init(&sm.bar[B_FULL + s], 1);
            mbar_init(&sm.bar[B_READY + s], 4);
            mbar_init(&sm.bar[B_DONE + s], 4);
        }
        mbar_init(&sm.bar[B_STATE], 4);
        mbar_init(&sm.bar[B_STATE1], 4);
        mbar_init(&sm.bar[B_X], 1);
        mbar_init(&sm.bar[B_G], 1);
        mbar_init(&sm.bar[B_GFREE], 4);
        mbar_init(&sm.bar[B_TD], 1);
        sm.abort_flag = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tm_q);
        tma_prefetch_desc(&tm_k);
        tma_prefetch_desc(&tm_v);
    }
    if (tid < 32) tmem_alloc(&sm.tmem, TM_COLS<D>);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // One block per SM: 384 threads x 168 registers at launch = 128 x (240 + 200 + 64).  Two: 384 x 80 = 128 x (152 + 64 + 24).
    if (tid < CHAIN_T) {
        if (BPS == 1) asm volatile("setmaxnreg.inc.sync.aligned.u32 240;");
        else asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
        chain<D, BPS, OUT>(p, sm, wk, nchunks);
    } else if (tid < CHAIN_T + PREP_T) {
        if (BPS == 1) asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
        else asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        prepare<D, BPS, VAR>(p, sm, wk, nchunks);
    } else {
        if (BPS == 1) asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        else asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");
        if (tid < CHAIN_T + PREP_T + 32) issue<D, BPS, !std::is_void<OUT>::value>(&tm_q, &tm_k, &tm_v, sm, wk, nchunks);
    }
    tc_fence_before();
    __syncthreads();
    if (sm.abort_flag) {   // copies and products issued just before a wait gave up finish first
        for (int i = 0; i < 32; ++i) __nanosleep(1000);
        if (tid == 0 && p.status_word) atomicExch(p.status_word, (int)KLA_ERR_TIMEOUT);
    }
    if (tid < 32) {
        tc_fence_after();
        tmem_dealloc(sm.tmem, TM_COLS<D>);
    }
}

// ---- host side: tensor maps and launch ---------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    });
    return fn;
}

// segment pass 1: (seg_G - 1) segments per sequence, twice the slices; p.n_seq counts all segments there
template <int D>
int blocks_of(const ChunkParams &p)
{
    return p.seg_pass == 1 ? (p.n_seq / p.seg_G) * (p.seg_G - 1) * p.H * 2 * (D / NS) : p.n_seq * p.H * (D / NS);
}
template <int D, int BPS, typename OUT, bool VAR>
cudaError_t launch_v(const ChunkParams &p, cudaStream_t stream)
{
    const uint64_t n_tok = (uint64_t)p.B * p.T;
    CUtensorMap tq, tk, tv;
    if (!make_tile_map(&tq, p.q, n_tok, (uint64_t)p.H * D) || !make_tile_map(&tk, p.k, n_tok, (uint64_t)p.H * D) ||
        !make_tile_map(&tv, p.v, n_tok, (uint64_t)p.H * D))
        return cudaErrorInvalidValue;
    auto kern = kla_chunk_mma_kernel<D, BPS, OUT, VAR>;
    const int smem = (int)sizeof(Smem<D, BPS>);
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (err != cudaSuccess) return err;
    const int grid = blocks_of<D>(p);
    if (grid == 0) return cudaSuccess;
    kern<<<grid, NT, smem, stream>>>(tq, tk, tv, p);
    count_launch(1);
    return cudaGetLastError();
}
template <int D, typename OUT>
cudaError_t launch_o(const ChunkParams &p, cudaStream_t stream)
{
    const bool var = (p.variant & ~VARIANT_WY) != 0;
    if constexpr (D == 64)
        if (blocks_of<D>(p) > sm_count()) return var ? launch_v<D, 2, OUT, true>(p, stream) : launch_v<D, 2, OUT, false>(p, stream);
    return var ? launch_v<D, 1, OUT, true>(p, stream) : launch_v<D, 1, OUT, false>(p, stream);
}
template <int D>
cudaError_t launch_d(const ChunkParams &p, int out_dtype, cudaStream_t stream)
{
    if (p.seg_pass == 1) return launch_o<D, void>(p, stream);
    return out_dtype == KLA_BF16 ? launch_o<D, __nv_bfloat16>(p, stream) : launch_o<D, float>(p, stream);
}

}  // namespace

bool make_tile_map(void *map, const void *base, uint64_t rows, uint64_t row_elems)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {row_elems, rows};
    cuuint64_t strides[1] = {row_elems * 2};
    cuuint32_t box[2] = {64, 64};
    cuuint32_t estr[2] = {1, 1};
    return fn(static_cast<CUtensorMap *>(map), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool chunk_tc_supported(int d, int chunk, int io_dtype)
{
    return (d == 64 || d == 128) && chunk == 64 && io_dtype == KLA_BF16;
}

cudaError_t launch_chunk_tc(const ChunkParams &p, int d, int io_dtype, int out_dtype, cudaStream_t stream)
{
    (void)io_dtype;
    if (d == 128 && (p.variant & VARIANT_WY)) return launch_chunk_wy(p, out_dtype, stream);
    return d == 128 ? launch_d<128>(p, out_dtype, stream) : launch_d<64>(p, out_dtype, stream);
}

}  // namespace kla
