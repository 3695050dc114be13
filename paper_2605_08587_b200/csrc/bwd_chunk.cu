// Reverse-mode derivative of the KLA recurrence, chunkwise (bf16 inputs).  The paper prints no backward; this is the derivative
// of its chunk algebra (Eqs. 7-9), which is the derivative of the recurrence of Algorithm 1 left up to the order of the sums.
//
// One chunk of 64 tokens, g the chunk-local running sum of log alpha, Gam = diag(exp g_i), D = diag(exp(g_C - g_j)), gC = exp g_C,
// A_ij = exp(g_i - g_j), X = A^- o K K^T, P = A o Q K^T, B = diag(beta), T = (I + B X)^-1:
//
//     forward     R = V - Gam K S_0,  U = T B R,  O = Gam Q S_0 + P U,  S_1 = gC S_0 + K^T D U
//     backward    dU = P^T dO + D K G_1,  w = T^T dU,  lam = B w (= dV),  G_0 = gC G_1 + (Gam Q)^T dO - (Gam K)^T lam
//     gradients   dQ = Gam dO S_0^T + F K,               F = A o (dO U^T), lower triangle
//                 dK = E K - Gam lam S_0^T               E = -A o (lam U^T), strictly lower   ("row" side: k_i as a query)
//                    + E^T K + F^T Q + D U G_1^T                                              ("column" side: k_j as a key)
//                    - 2 k dbeta beta / n,  deta = dbeta / n (Eq. 3),  dbeta_i = sum (U / beta)_i o w_i
//     decay       exp(g_i) multiplies q_i and the row side of k_i, exp(-g_j) the column side of k_j, so
//                 dg_i = q_i . dq_i + k_i . dk_i(row) - k_i . dk_i(column), dg_C += <G_1, S_1>, dlog_alpha_t = sum_{i >= t} dg_i
//
// (G = dL/dS.)  Three launches:
//   1. prepare   one block per (chunk, head): decays, beta, T (as operand planes), P^T dO, per-token scalars;
//   2. chains    one block per (sequence, head, 64 columns) and direction: the recurrences over S and over G, each leaving the
//                state at every chunk (and U, respectively dV) in the workspace; the two do not depend on each other;
//   3. gradients one block per (chunk, head): everything that is left, in parallel over chunks.
// Token by token on CUDA cores (bwd_scan.cu, which stays for fp32 inputs) the layer shape took 8.1 ms.
//
// Precision.  mma.sync truncates its fp32 sums (mma_pieces.cuh), so how often a sum is truncated at its full size decides how exact it is.
// The products of the first planes, the size of the result, are therefore summed apart from the terms of the lower planes (2^-8 of it
// and less), in runs of at most eight, and everything else is added in fp32: the states to what a chunk adds to them, the two halves
// of a long sum, the parts of a gradient.  2-norm errors against fp64, B 8, H 8, T 4096, d 128: dq 1.4e-7, dk 1.5e-7, dv 1.4e-7,
// dlog_alpha 3.4e-7, deta 1.9e-7, dinit 1.5e-7, as those of the token-by-token kernel (1.8e-7, 1.9e-7, 1.9e-7, 2.9e-7, 2.0e-7, 1.9e-7);
// with all terms in one accumulator they were 4e-7 .. 1.1e-6.  Cost when it was built: 1.50 -> 1.62 ms.
//
// beta = 0 (eta = 0) would make U = B (...) carry no trace of the residual e = U / beta that dbeta needs; such a beta is taken
// as 1e-30, where every gradient has its limit to the last bit.
#include <cuda.h>

#include "common.cuh"
#include "mma_pieces.cuh"
#include "scan_pieces.cuh"
#include "solve_pieces.cuh"
#include "umma.cuh"

namespace kla {

namespace {

using namespace wmm;

constexpr int C = 64;        // chunk length
constexpr int T_BYTES = 3 * 8192;   // three planes of a 64 x 64 operand

// Per-token scalars of one chunk, as the kernels hand them on.
struct Scal {
    float beta[C];   // Eq. 3 (or eta), tokens past the end: 0; never 0 otherwise
    float gam[C];    // exp(g_i)
    float dec[C];    // exp(g_C - g_i)
    float g2h[C], g2l[C];   // log2(e) g_i = g2h + g2l (differences of large sums keep their fp32 digits)
    float nrm[C];    // ||k||^2 + eps
    float qinv[C];   // 1 / ||q|| with the normalised read-out, else 1
    float dn[C];     // used by the gradients: dk_i += dn_i k_i through the norm in Eq. 3
};

struct BwdChunkParams {
    const __nv_bfloat16 *q, *k, *v, *dout;
    const float *log_alpha, *eta;
    const float *init_state, *dfinal;
    float *dq, *dk, *dv, *dlog_alpha, *deta, *dinit;
    const int32_t *cu_seqlens;   // null: fixed length T
    const int32_t *order;        // packed input: sequences longest first (or null)
    int32_t T, H, n_seq;
    float eps;
    int32_t coeff_eta, qnorm;
    // workspace, one entry per (slot, head); a slot is a chunk: n ceil(T / 64) + c, packed tok0 / 64 + n + c
    unsigned char *tpl;   // T as three operand planes, 64 x 64 each, sw128 layout
    float *pdo;           // (P^T dO)^T  [D / 16][8] accumulator tiles
    float *s0, *g1;       // S_0^T, G_1^T  d 64: [d_v / 16][d_k / 8] accumulator tiles; d 128: [d_v][d_k]
    float *u;             // U           [64][D]
    Scal *scal;
    int32_t n_slots;
    int32_t test_timeout;
    int32_t *status_word;
};
// How states and P^T dO cross the workspace.  An accumulator tile is 16 rows x 8 columns with a lane's four values side by side: a warp
// of the chains then writes and reads 512 bytes in a row, where rows take 8 lines to an instruction.  The gradients' planes are rows,
// and from tiles a thread has two neighbours to write to them (4-byte stores), from rows eight (16 bytes).  Measured, us:
//                                       chains    gradients   the call
//     d 64, 16 packed sequences         406 -> 354   778 -> 778   1433 -> 1379    states as rows -> as tiles
//     d 128, B 8, H 8, T 4096           563 -> 566   813 -> 835   1498 -> 1527
// so the states are tiles at d 64 alone (at d 128 a chunk has more products to cover its stores with, and the gradients spill registers
// with tiles, 20 bytes each way, where with rows they do not).  P^T dO, which only the chains read, is tiles at both (1443 -> 1433, 1513 -> 1498).
template <int D>
constexpr bool STATE_TILES = D == 64;
struct TileMaps {
    CUtensorMap q, k, v, dout;   // 64 tokens x 64 columns
};

struct Where {
    int n, c, tok0, len;   // sequence, chunk of it, its first token, its length
};
__device__ __forceinline__ int slot_of(const BwdChunkParams &p, int n, int tok0, int c)
{
    return p.cu_seqlens ? tok0 / C + n + c : n * ((p.T + C - 1) / C) + c;
}
// The chunk of a slot; c beyond the sequence's chunks: the slot is empty.
__device__ __forceinline__ Where locate(const BwdChunkParams &p, int slot)
{
    Where w;
    if (!p.cu_seqlens) {
        const int cps = (p.T + C - 1) / C;
        w.n = slot / cps;
        w.c = slot - w.n * cps;
        w.tok0 = w.n * p.T;
        w.len = p.T;
        return w;
    }
    int lo = 0, hi = p.n_seq - 1;   // last n with cu[n] / 64 + n <= slot (strictly increasing in n)
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.cu_seqlens[mid] / C + mid <= slot) lo = mid;
        else hi = mid - 1;
    }
    w.n = lo;
    w.tok0 = p.cu_seqlens[lo];
    w.len = p.cu_seqlens[lo + 1] - w.tok0;
    w.c = slot - (w.tok0 / C + lo);
    return w;
}

// `bytes` (a multiple of 16, from a 16-byte boundary) on their way into L2.
__device__ __forceinline__ void prefetch_l2(const void *x, int bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(x), "r"(bytes) : "memory");
}

// Rows t0 .. t0 + 63 (of which `rows` exist, the others become zero) of a [token][H][D] array, columns col .. col + 64 NB - 1
// of head h, into NB consecutive 64 x 64 tiles; all NTH threads.
template <int NB, int D, int NTH>
__device__ __forceinline__ void load_tile(uint32_t dst, const __nv_bfloat16 *src, size_t t0, int rows, int H, int h, int col, int tid)
{
#pragma unroll
    for (int e = tid; e < NB * C * 8; e += NTH) {
        const int r = e / (NB * 8), ch = e % (NB * 8);
        const int rr = r < rows ? r : 0;
        cp16(dst + (ch >> 3) * 8192 + sw128(r, ch & 7), src + ((t0 + rr) * H + h) * D + col + ch * 8, r < rows);
    }
}

// ---- 1. prepare -----------------------------------------------------------------------------------------------------------
template <int D>
struct PrepSmem {
    union {
        struct {
            alignas(1024) unsigned char k[D / 64 * 8192], q[D / 64 * 8192];
        };
        alignas(1024) unsigned char p[T_BYTES];   // P, three planes, once K and Q have been read
        alignas(16) float mm[32 * LDM];           // scratch of the inverse, once P^T dO is done
    };
    alignas(1024) unsigned char dout[D / 64 * 8192];
    alignas(16) float tl[C * LDT];            // X, overwritten by T
    Scal s;
    float eta[C];
};

// What bounds it: the latency of its phases (the levels of the inverse, each behind barriers), so blocks per SM: P over K and Q
// gives room for a third one (B 8, H 8, T 4096, d 128: 198 -> 168 us; 16 packed sequences, d 64: 369 -> 305 us).  At d 64, with the
// scratch of the inverse over P as well, a fourth fits and 64 registers hold everything (-27 us).
template <int D>
__global__ void __launch_bounds__(256, D == 64 ? 4 : 3) kla_bwd_prepare_kernel(BwdChunkParams p)
{
    extern __shared__ __align__(1024) unsigned char smem_dyn[];   // used as declared: rounded up at run time, every access would be generic
    using Smem = PrepSmem<D>;
    Smem &sm = *reinterpret_cast<Smem *>(smem_dyn);
    constexpr int NB = D / 64;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int slot = blockIdx.x / p.H, h = blockIdx.x % p.H;
    const Where w = locate(p, slot);
    if (w.c * C >= w.len) return;
    const int rows = min(C, w.len - w.c * C);
    const size_t t0 = (size_t)w.tok0 + w.c * C;
    load_tile<NB, D, 256>(smem_u32(sm.k), p.k, t0, rows, p.H, h, 0, tid);
    load_tile<NB, D, 256>(smem_u32(sm.q), p.q, t0, rows, p.H, h, 0, tid);
    cp_commit();
    load_tile<NB, D, 256>(smem_u32(sm.dout), p.dout, t0, rows, p.H, h, 0, tid);
    cp_commit();

    if (warp == 0) {   // decay sums in fp64 (tokens 2 lane, 2 lane + 1)
        const int a = 2 * lane;
        const double x0 = a < rows ? (double)p.log_alpha[(t0 + a) * p.H + h] : 0.0;
        const double x1 = a + 1 < rows ? (double)p.log_alpha[(t0 + a + 1) * p.H + h] : 0.0;
        double incl = x0 + x1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const double gc = __shfl_sync(0xffffffffu, incl, 31);
        const double g[2] = {incl - x1, incl};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            sm.s.gam[a + u] = expf((float)g[u]);
            sm.s.dec[a + u] = expf((float)(gc - g[u]));
            const double g2 = g[u] * 1.4426950408889634074;
            sm.s.g2h[a + u] = (float)g2;
            sm.s.g2l[a + u] = (float)(g2 - (double)(float)g2);
        }
    } else if (warp < 3) {
        const int i = (warp - 1) * 32 + lane;
        sm.eta[i] = i < rows ? p.eta[(t0 + i) * p.H + h] : 0.f;
        sm.s.qinv[i] = 1.f;
        sm.s.dn[i] = 0.f;
    }
    for (int e = tid; e < C * LDT; e += 256) sm.tl[e] = 0.f;
    cp_wait<1>();
    __syncthreads();
    if (p.qnorm && tid < C) {
        float n = 0.f;
        for (int e = 0; e < NB * 8; ++e) {
            const uint4 raw = *reinterpret_cast<const uint4 *>(sm.q + (e >> 3) * 8192 + sw128(tid, e & 7));
            const uint32_t x[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 f = unpack(x[u]);
                n += f.x * f.x + f.y * f.y;
            }
        }
        sm.s.qinv[tid] = tid < rows ? 1.f / sqrtf(n) : 0.f;
    }

    // K K^T (warps 0..3) and Q K^T (warps 4..7): 16 rows each, columns up to the diagonal block
    const int mt = warp & 3, i0 = mt * 16;
    float acc[8][4];
#pragma unroll
    for (int t = 0; t < 8; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[t][e] = 0.f;
    {
        const uint32_t at = smem_u32(warp < 4 ? sm.k : sm.q), bt = smem_u32(sm.k);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
            const uint32_t off = (ks >> 2) * 8192;
            uint32_t a[4];
            frag_a(a, at + off, i0, (ks & 3) * 16, lane);
#pragma unroll
            for (int np = 0; np < 4; ++np) {
                if (np <= mt) {
                    uint32_t b[4];
                    frag_b(b, bt + off, (ks & 3) * 16, np * 16, lane);
                    mma(acc[2 * np], a, b[0], b[1]);
                    mma(acc[2 * np + 1], a, b[2], b[3]);
                }
            }
        }
    }
    // accumulator element (t, e): row i0 + lane / 4 (+ 8 for e >= 2), column 8 t + 2 (lane % 4) + (e & 1)
    const int r0 = i0 + (lane >> 2), cq = 2 * (lane & 3);
    if (warp < 4) {
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = r0 + (e >> 1) * 8, j = 8 * t + cq + (e & 1);
                if (i == j) {   // ||k_i||^2
                    const float n = acc[t][e] + p.eps;
                    float b = i < rows ? (p.coeff_eta ? sm.eta[i] : sm.eta[i] / n) : 0.f;
                    if (i < rows && fabsf(b) < 1e-30f) b = 1e-30f;
                    sm.s.nrm[i] = n;
                    sm.s.beta[i] = b;
                }
            }
    }
    __syncthreads();   // scalars are complete
    if (warp < 4) {
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = r0 + (e >> 1) * 8, j = 8 * t + cq + (e & 1);
                if (j < i) sm.tl[i * LDT + j] = exp2f((sm.s.g2h[i] - sm.s.g2h[j]) + (sm.s.g2l[i] - sm.s.g2l[j])) * acc[t][e];
            }
    } else {
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                const int i = r0 + (e >> 1) * 8, j = 8 * t + cq;
                const float hi = sm.s.g2h[i], li = sm.s.g2l[i], qi = sm.s.qinv[i];
                const float x = j <= i ? qi * exp2f((hi - sm.s.g2h[j]) + (li - sm.s.g2l[j])) * acc[t][e] : 0.f;
                const float y = j + 1 <= i ? qi * exp2f((hi - sm.s.g2h[j + 1]) + (li - sm.s.g2l[j + 1])) * acc[t][e + 1] : 0.f;
                uint32_t a, b, c;
                split3(x, y, a, b, c);
                const uint32_t off = sw128(i, t) + 4 * (lane & 3);
                *reinterpret_cast<uint32_t *>(sm.p + off) = a;
                *reinterpret_cast<uint32_t *>(sm.p + 8192 + off) = b;
                *reinterpret_cast<uint32_t *>(sm.p + 16384 + off) = c;
            }
    }
    cp_wait<0>();
    __syncthreads();
    const size_t ch = (size_t)slot * p.H + h;
    if (tid < sizeof(Scal) / 16) reinterpret_cast<float4 *>(p.scal + ch)[tid] = reinterpret_cast<const float4 *>(&sm.s)[tid];

    // (P^T dO)^T = dO^T P: 16 rows (columns of V) per warp
    if (warp * 16 < D) {
        float o[8][4];
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[t][e] = 0.f;
        const uint32_t at = smem_u32(sm.dout) + (warp >> 2) * 8192, bt = smem_u32(sm.p);
#pragma unroll
        for (int pl = 2; pl >= 0; --pl)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                uint32_t a[4];
                frag_at(a, at, (warp & 3) * 16, ks * 16, lane);
#pragma unroll
                for (int np = 0; np <= ks; ++np) {
                    uint32_t b[4];
                    frag_bt(b, bt + pl * 8192, ks * 16, np * 16, lane);
                    mma(o[2 * np], a, b[0], b[1]);
                    mma(o[2 * np + 1], a, b[2], b[3]);
                }
            }
        float *dst = p.pdo + ch * D * C + warp * 16 * C + lane * 4;
#pragma unroll
        for (int t = 0; t < 8; ++t) store4(dst + 128 * t, make_float4(o[t][0], o[t][1], o[t][2], o[t][3]));
    }

    // T = (I + B X)^-1: 8 x 8 diagonal blocks by substitution (column tid % 8 of block tid / 8), then block merges
    const float *bet = sm.s.beta;
    float x[8];
    if (tid < 64) {
        const int blk = tid >> 3, j = tid & 7;
        const float *Lb = sm.tl + (blk * 8) * LDT + blk * 8;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            float s = 0.f;
#pragma unroll
            for (int m = 0; m < r; ++m) s += Lb[r * LDT + m] * x[m];
            x[r] = (r == j) ? 1.f : ((r > j) ? -bet[blk * 8 + r] * s : 0.f);
        }
    }
    __syncthreads();
    if (tid < 64) {
        const int blk = tid >> 3, j = tid & 7;
#pragma unroll
        for (int r = 0; r < 8; ++r) sm.tl[(blk * 8 + r) * LDT + blk * 8 + j] = x[r];
    }
    __syncthreads();
    // (a block whose rows all lie past the end of the sequence is zero as it stands)
    if (rows > 8) merge_level<8, LDM, false>(sm.tl, sm.mm, bet, tid, [] { __syncthreads(); });
    if (rows > 16) merge_level<16, LDM, false>(sm.tl, sm.mm, bet, tid, [] { __syncthreads(); });
    if (rows > 32) merge_level<32, LDM, false>(sm.tl, sm.mm, bet, tid, [] { __syncthreads(); });
    // T as three operand planes: 8 columns per item
    unsigned char *tp = p.tpl + ch * T_BYTES;
#pragma unroll
    for (int e = tid; e < C * 8; e += 256) {
        const int r = e >> 3, c8 = e & 7;
        uint32_t hh[4], mm[4], ll[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) split3(sm.tl[r * LDT + c8 * 8 + 2 * u], sm.tl[r * LDT + c8 * 8 + 2 * u + 1], hh[u], mm[u], ll[u]);
        const uint32_t off = sw128(r, c8);
        *reinterpret_cast<uint4 *>(tp + off) = make_uint4(hh[0], hh[1], hh[2], hh[3]);
        *reinterpret_cast<uint4 *>(tp + 8192 + off) = make_uint4(mm[0], mm[1], mm[2], mm[3]);
        *reinterpret_cast<uint4 *>(tp + 16384 + off) = make_uint4(ll[0], ll[1], ll[2], ll[3]);
    }
}

// ---- 2. chains ------------------------------------------------------------------------------------------------------------
// Four warps, 16 columns of d_v each; the transposed state (16 x D) stays in registers as accumulator tiles, is split into
// operand planes on the fly and never leaves the warp.  K is fetched a chunk ahead into the other of two buffers; what a chunk
// uses last (T, V, respectively T, Q, dO) has one buffer and is fetched as soon as every warp has passed it.  One thread fetches
// by TMA: as asynchronous copies of 16 bytes the 33 of a thread and chunk, a dozen instructions each that run once and come from
// beyond the instruction caches, took 2 900 (backward) and 1 200 (forward) cycles of a chunk's 16 300 and 13 000.
// What bounds it: the latency of one warp per scheduler and block, which issues in order.  Its 504 (forward) and 696 (backward)
// instructions of the warp-level tensor pipe per chunk at D = 128 keep that pipe busy for 56 % of the cycles.
// Both directions are one launch so that an SM holds a block of each and one fills the other's latencies.
template <int D>
struct ChainSmem {
    alignas(1024) unsigned char k[2][D / 64 * 8192];
    alignas(1024) unsigned char t[T_BYTES];
    alignas(1024) unsigned char vd[8192];            // V (forward), dO (backward): this block's 64 columns
    alignas(1024) unsigned char q[D / 64 * 8192];    // backward only
    Scal s[2];
    alignas(8) uint64_t bar[2];                      // K, scalars, T (and V) of a chunk; Q and dO of it
};
constexpr long long CHAIN_WAIT_LIMIT = 2000000000LL;   // SM clocks (~1 s) before a wait gives up

// Rows from `rows` on of NB 64 x 64 tiles, which hold what follows the sequence, become zero.
template <int NB>
__device__ __forceinline__ void zero_rows(unsigned char *tile, int rows, int tid)
{
#pragma unroll 1
    for (int e = tid; e < (C - rows) * 8 * NB; e += 128) {
        const int r = rows + e / (8 * NB), ch = e % (8 * NB);
        *reinterpret_cast<uint4 *>(tile + (ch >> 3) * 8192 + sw128(r, ch & 7)) = make_uint4(0, 0, 0, 0);
    }
}

// acc[token tile] = (16 x D state) (64 x D tile)^T: columns are tokens.  `late`: called before the last products
template <int D, typename F>
__device__ __forceinline__ void state_times_tile(float (&acc)[8][4], const float (&S)[D / 8][4], uint32_t kt, int lane, F &&late)
{
    float low[8][4];
#pragma unroll
    for (int t = 0; t < 8; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[t][e] = low[t][e] = 0.f;
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
        if (ks == D / 16 - 2) late();
        uint32_t a[3][4];
        split_a(S[2 * ks], S[2 * ks + 1], a[0], a[1], a[2]);
        uint32_t b[4][4];
#pragma unroll
        for (int np = 0; np < 4; ++np) frag_b(b[np], kt + (ks >> 2) * 8192, (ks & 3) * 16, np * 16, lane);
#pragma unroll
        for (int pl = 0; pl < 3; ++pl)
#pragma unroll
            for (int np = 0; np < 4; ++np) {
                mma(pl ? low[2 * np] : acc[2 * np], a[pl], b[np][0], b[np][1]);
                mma(pl ? low[2 * np + 1] : acc[2 * np + 1], a[pl], b[np][2], b[np][3]);
            }
    }
#pragma unroll
    for (int t = 0; t < 8; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[t][e] += low[t][e];
}
// S = gc S + (64 tokens of a 16 x 64 factor, three planes) (tile)[those tokens][D]
template <int D>
__device__ __forceinline__ void state_update(float (&S)[D / 8][4], float gc, const uint32_t (&a)[4][3][4], uint32_t tile, int lane)
{
#pragma unroll
    for (int np = 0; np < D / 16; ++np) {
        uint32_t b[4][4];
        float d[2][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) d[0][e] = d[1][e] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) frag_bt(b[ks], tile + (np >> 2) * 8192, ks * 16, (np & 3) * 16, lane);
#pragma unroll
        for (int pl = 2; pl >= 0; --pl)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                mma(d[0], a[ks][pl], b[ks][0], b[ks][1]);
                mma(d[1], a[ks][pl], b[ks][2], b[ks][3]);
            }
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) S[2 * np + t][e] = gc * S[2 * np + t][e] + d[t][e];
    }
}
// three-plane x three-plane product on two tiles, terms down to 2^-24: all but the first
__device__ __forceinline__ void mma5(float (&c0)[4], float (&c1)[4], const uint32_t (&a)[3][4], const uint32_t (&b)[3][4])
{
    constexpr int PA[5] = {1, 2, 0, 1, 0}, PB[5] = {1, 0, 2, 0, 1};
#pragma unroll
    for (int t = 0; t < 5; ++t) {
        mma(c0, a[PA[t]], b[PB[t]][0], b[PB[t]][1]);
        mma(c1, a[PA[t]], b[PB[t]][2], b[PB[t]][3]);
    }
}

template <int D, bool BWD>
__device__ __forceinline__ void chain(const BwdChunkParams &p, const TileMaps &tm, ChainSmem<D> &sm, int unit)
{
    constexpr int NB = D / 64;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sl = unit % NB, h = (unit / NB) % p.H;
    int n = unit / (NB * p.H);
    if (p.order) n = p.order[n];
    int tok0, len;
    if (p.cu_seqlens) {
        tok0 = p.cu_seqlens[n];
        len = p.cu_seqlens[n + 1] - tok0;
    } else {
        tok0 = n * p.T;
        len = p.T;
    }
    const int nc = (len + C - 1) / C;
    const int r = lane >> 2, cq = 2 * (lane & 3);
    const int col = sl * 64 + warp * 16 + r;   // columns col, col + 8 of d_v
    // element (t, e) of a state tile: column col (+ 8 for e >= 2), row 8 t + cq + (e & 1)
    float S[D / 8][4];
    {
        const float *src = BWD ? p.dfinal : p.init_state;
        const size_t base = ((size_t)n * p.H + h) * D * D + col;
#pragma unroll
        for (int t = 0; t < D / 8; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) S[t][e] = src ? src[base + (size_t)(8 * t + cq + (e & 1)) * D + (e >> 1) * 8] : 0.f;
    }
    const size_t ch0 = (size_t)slot_of(p, n, tok0, 0) * p.H + h;   // chunk c: + c H
    auto rows_of = [&](int c) { return min(C, len - c * C); };
    // (one thread)
    auto load_k = [&](int c) {
        umma::mbar_expect_tx(&sm.bar[0], NB * 8192 + sizeof(Scal) + T_BYTES + (BWD ? 0 : 8192));
#pragma unroll
        for (int b = 0; b < NB; ++b) umma::tma_load_2d(sm.k[c & 1] + b * 8192, &tm.k, h * D + b * 64, tok0 + c * C, &sm.bar[0]);
        umma::bulk_load(&sm.s[c & 1], p.scal + ch0 + (size_t)c * p.H, sizeof(Scal), &sm.bar[0]);
    };
    auto load_t = [&](int c) {   // counted with K
        umma::bulk_load(sm.t, p.tpl + (ch0 + (size_t)c * p.H) * T_BYTES, T_BYTES, &sm.bar[0]);
        if (!BWD) umma::tma_load_2d(sm.vd, &tm.v, h * D + sl * 64, tok0 + c * C, &sm.bar[0]);
    };
    auto load_q = [&](int c) {
        umma::mbar_expect_tx(&sm.bar[1], (NB + 1) * 8192);
        umma::tma_load_2d(sm.vd, &tm.dout, h * D + sl * 64, tok0 + c * C, &sm.bar[1]);
#pragma unroll
        for (int b = 0; b < NB; ++b) umma::tma_load_2d(sm.q + b * 8192, &tm.q, h * D + b * 64, tok0 + c * C, &sm.bar[1]);
    };
    if (tid == 0) {
        umma::mbar_init(&sm.bar[0], 1);
        umma::mbar_init(&sm.bar[1], 1);
        umma::mbar_fence_init();
    }
    __syncthreads();
    bool late = false;   // a wait ran out (for the whole block)
    const int step = BWD ? -1 : 1;
    int c = BWD ? nc - 1 : 0;
    // (test hook: T and V, in the backward direction Q and dO, are never asked for, and the wait for them runs out)
    if (nc > 0 && tid == 0) {
        load_k(c);
        if (BWD || !p.test_timeout) load_t(c);
    }
    for (int it = 0; it < nc; ++it, c += step) {
        const Scal &s = sm.s[c & 1];
        const size_t ch = ch0 + (size_t)c * p.H;
        const uint32_t kt = smem_u32(sm.k[c & 1]), tt = smem_u32(sm.t);
        const int rows = rows_of(c);
        late = __syncthreads_or(!umma::mbar_wait(&sm.bar[0], it & 1, CHAIN_WAIT_LIMIT));
        if (late) break;
        if (rows < C) {
            zero_rows<NB>(sm.k[c & 1], rows, tid);
            if (!BWD) zero_rows<1>(sm.vd, rows, tid);
            umma::fence_async_smem();
            __syncthreads();
        }
        if (tid == 0) {
            if (BWD && !p.test_timeout) load_q(c);
            if (it + 1 < nc) {   // (P^T dO: 1 431 -> 1 380 us with 16 packed sequences, d 64)
                load_k(c + step);
                if (BWD) prefetch_l2(p.pdo + (ch0 + (size_t)(c + step) * p.H) * D * C + sl * 64 * C, 64 * C * 4);
            }
        }
        // the state at this end of the chunk, transposed
        {
            float *dst = (BWD ? p.g1 : p.s0) + ch * D * D;
            if constexpr (STATE_TILES<D>) {
                dst += (sl * 4 + warp) * 16 * D + lane * 4;
#pragma unroll
                for (int t = 0; t < D / 8; ++t) store4(dst + 128 * t, make_float4(S[t][0], S[t][1], S[t][2], S[t][3]));
            } else {
                dst += (size_t)col * D + cq;
#pragma unroll
                for (int t = 0; t < D / 8; ++t) {
                    store2(dst + 8 * t, S[t][0], S[t][1]);
                    store2(dst + 8 * D + 8 * t, S[t][2], S[t][3]);
                }
            }
        }
        float4 pd[BWD ? 8 : 1];
        float x[8][4], y[8][4];
        state_times_tile<D>(x, S, kt, lane, [&] {   // (K S_0)^T or (K G_1)^T
            if constexpr (BWD) {
                const float *src = p.pdo + ch * D * C + (sl * 4 + warp) * 16 * C + lane * 4;
#pragma unroll
                for (int t = 0; t < 8; ++t) pd[t] = load4(src + 128 * t);
            }
        });
        if constexpr (BWD) {   // dU = D K G_1 + P^T dO
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const float2 d = *reinterpret_cast<const float2 *>(&s.dec[8 * t + cq]);
                x[t][0] = d.x * x[t][0] + pd[t].x;
                x[t][1] = d.y * x[t][1] + pd[t].y;
                x[t][2] = d.x * x[t][2] + pd[t].z;
                x[t][3] = d.y * x[t][3] + pd[t].w;
            }
        } else {   // B (V - Gam K S_0)
#pragma unroll
            for (int tp = 0; tp < 4; ++tp) {
                uint32_t vv[4];
                ldsm4t(vv, smem_u32(sm.vd) + sw128(tp * 16 + (lane & 7) + (lane >> 4) * 8, warp * 2 + ((lane >> 3) & 1)));
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int t = 2 * tp + u;
                    const float2 b = *reinterpret_cast<const float2 *>(&s.beta[8 * t + cq]), g = *reinterpret_cast<const float2 *>(&s.gam[8 * t + cq]);
                    const float2 v0 = unpack(vv[2 * u]), v1 = unpack(vv[2 * u + 1]);
                    x[t][0] = b.x * (v0.x - g.x * x[t][0]);
                    x[t][1] = b.y * (v0.y - g.y * x[t][1]);
                    x[t][2] = b.x * (v1.x - g.x * x[t][2]);
                    x[t][3] = b.y * (v1.y - g.y * x[t][3]);
                }
            }
        }
        // U^T = rhs^T T^T (T_ij, j <= i) or w^T = dU^T T
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) y[t][e] = 0.f;
        uint32_t xh[4][4];
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            uint32_t a[3][4];
            split_a(x[2 * ks], x[2 * ks + 1], a[0], a[1], a[2]);
#pragma unroll
            for (int e = 0; e < 4; ++e) xh[ks][e] = a[0][e];
#pragma unroll
            for (int np = BWD ? 0 : ks; np <= (BWD ? ks : 3); ++np) {
                uint32_t b[3][4];
#pragma unroll
                for (int pl = 0; pl < 3; ++pl) {
                    if (BWD) frag_bt(b[pl], tt + pl * 8192, ks * 16, np * 16, lane);
                    else frag_b(b[pl], tt + pl * 8192, ks * 16, np * 16, lane);
                }
                mma5(y[2 * np], y[2 * np + 1], a, b);
            }
        }
        // the first planes, 32 tokens at a time, added in fp32
#pragma unroll
        for (int half = 0; half < 2; ++half)
#pragma unroll
            for (int np = 0; np < 4; ++np) {
                if (BWD ? np > 2 * half + 1 : np < 2 * half) continue;
                float d[2][4];
#pragma unroll
                for (int e = 0; e < 4; ++e) d[0][e] = d[1][e] = 0.f;
#pragma unroll
                for (int ks = 2 * half; ks < 2 * half + 2; ++ks) {
                    if (BWD ? np > ks : np < ks) continue;
                    uint32_t b[4];
                    if (BWD) frag_bt(b, tt, ks * 16, np * 16, lane);
                    else frag_b(b, tt, ks * 16, np * 16, lane);
                    mma(d[0], xh[ks], b[0], b[1]);
                    mma(d[1], xh[ks], b[2], b[3]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) y[2 * np][e] += d[0][e], y[2 * np + 1][e] += d[1][e];
            }
        // every warp is done with T (and V); Q and dO have landed
        late = __syncthreads_or(BWD && !umma::mbar_wait(&sm.bar[1], it & 1, CHAIN_WAIT_LIMIT));
        if (late) break;
        if (BWD && rows < C) {
            zero_rows<NB>(sm.q, rows, tid);
            zero_rows<1>(sm.vd, rows, tid);
            umma::fence_async_smem();
            __syncthreads();
        }
        if (tid == 0 && it + 1 < nc) load_t(c + step);
        const float gc = s.gam[C - 1];
        if constexpr (BWD) {   // lam = B w
            float *dst = p.dv + (((size_t)tok0 + c * C + cq) * p.H + h) * D + col;
            const size_t row = (size_t)p.H * D;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const float2 b = *reinterpret_cast<const float2 *>(&s.beta[8 * t + cq]), g = *reinterpret_cast<const float2 *>(&s.gam[8 * t + cq]);
                y[t][0] *= b.x; y[t][1] *= b.y; y[t][2] *= b.x; y[t][3] *= b.y;
                if (8 * t + cq < rows) {
                    dst[(8 * t) * row] = y[t][0];
                    dst[(8 * t) * row + 8] = y[t][2];
                }
                if (8 * t + cq + 1 < rows) {
                    dst[(8 * t + 1) * row] = y[t][1];
                    dst[(8 * t + 1) * row + 8] = y[t][3];
                }
                y[t][0] *= -g.x; y[t][1] *= -g.y; y[t][2] *= -g.x; y[t][3] *= -g.y;
            }
        } else {
            float *dst = p.u + ch * C * D + (size_t)cq * D + col;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const float2 d = *reinterpret_cast<const float2 *>(&s.dec[8 * t + cq]);
                dst[(8 * t) * D] = y[t][0];
                dst[(8 * t) * D + 8] = y[t][2];
                dst[(8 * t + 1) * D] = y[t][1];
                dst[(8 * t + 1) * D + 8] = y[t][3];
                y[t][0] *= d.x; y[t][1] *= d.y; y[t][2] *= d.x; y[t][3] *= d.y;
            }
        }
        uint32_t a[4][3][4];
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) split_a(y[2 * ks], y[2 * ks + 1], a[ks][0], a[ks][1], a[ks][2]);
        state_update<D>(S, gc, a, kt, lane);   // += (D U)^T K, or -= (Gam lam)^T K
        if constexpr (BWD) {   // += dO^T (Gam Q): the decay goes with dO, in registers
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                uint32_t d[4];
                frag_at(d, smem_u32(sm.vd), warp * 16, ks * 16, lane);
                // registers: (row r, tokens cq, cq + 1), (row r + 8, ...), then tokens + 8
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int tk = ks * 16 + cq + (e >> 1) * 8;
                    const float2 f = unpack(d[e]), g = *reinterpret_cast<const float2 *>(&s.gam[tk]), qi = *reinterpret_cast<const float2 *>(&s.qinv[tk]);
                    split3(f.x * (g.x * qi.x), f.y * (g.y * qi.y), a[ks][0][e], a[ks][1][e], a[ks][2][e]);
                }
            }
            state_update<D>(S, 1.f, a, smem_u32(sm.q), lane);
        }
    }
    if (late) {   // copies issued just before a wait gave up finish first
        for (int i = 0; i < 32; ++i) __nanosleep(1000);
        if (tid == 0 && p.status_word) atomicExch(p.status_word, (int)KLA_ERR_TIMEOUT);
        return;
    }
    if (BWD && p.dinit) {
        float *dst = p.dinit + ((size_t)n * p.H + h) * D * D + col;
#pragma unroll
        for (int t = 0; t < D / 8; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) dst[(size_t)(8 * t + cq + (e & 1)) * D + (e >> 1) * 8] = S[t][e];
    }
}

template <int D>
__global__ void __launch_bounds__(128, 2) kla_bwd_chain_kernel(const __grid_constant__ TileMaps tm, BwdChunkParams p, int n_units)
{
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    ChainSmem<D> &sm = *reinterpret_cast<ChainSmem<D> *>(smem_dyn);
    // TMA permutes the pieces of a row by their address, ldmatrix here by their place in the tile: the same from a 1024-byte boundary on.
    // There is no static shared memory, so the tiles start on one; checked all the same.
    if (smem_u32(smem_dyn) & 1023) {
        if (threadIdx.x == 0 && p.status_word) atomicExch(p.status_word, (int)KLA_ERR_ALIGN);
        return;
    }
    // the backward chains, the longer ones, first
    if ((int)blockIdx.x < n_units) chain<D, true>(p, tm, sm, blockIdx.x);
    else chain<D, false>(p, tm, sm, blockIdx.x - n_units);
}

// ---- 3. gradients ---------------------------------------------------------------------------------------------------------
// One block of sixteen warps per (chunk, head).  Output columns (d_k) are taken in halves of 64: the operand planes of S_0, then
// of G_1, of one half share a buffer.  A warp owns 16 tokens x 16 columns; operands that two products have in common are
// loaded once for both.  Global loads of the next operand are requested before the products of the one at hand.
constexpr int GW = 16;         // warps
constexpr int GT = 32 * GW;
template <int D>
struct GradSmem {
    unsigned char dout[D / 64 * 8192];            // [token][d_v]
    unsigned char u[D / 64 * T_BYTES];            // planes, [token][d_v] (plane pl, block b at (pl NB + b) 8192)
    unsigned char lam[D / 64 * T_BYTES];
    unsigned char f[T_BYTES], e[T_BYTES];         // planes, [i][j]; only blocks on and below the diagonal are used
    unsigned char sg[3 * D * 128];                // S_0^T or G_1^T, planes, [d_v][64 of d_k]
    unsigned char k[8192], q[8192];               // [token][64 of d_k]
    Scal s;
    float red[4][64];                             // dg_i, the parts of the four column groups of the warps
};

// Asks for what block `b` of the gradients reads to be brought into L2; nothing is waited for.  Called for the block that will
// follow on this SM: its first loads then do not go to DRAM (B 8, H 8, T 4096, d 128: 1 614 -> 1 590 us for the whole call).
template <int D>
__device__ __forceinline__ void prefetch_block(const BwdChunkParams &p, int b, int tid)
{
    const int slot = b / p.H, h = b % p.H;
    const Where w = locate(p, slot);
    if (w.c * C >= w.len) return;
    const int rows = min(C, w.len - w.c * C);
    const size_t t0 = (size_t)w.tok0 + w.c * C, ch = (size_t)slot * p.H + h;
    if (tid == 0) {
        prefetch_l2(p.u + ch * C * D, C * D * 4);
        prefetch_l2(p.s0 + ch * D * D, D * D * 4);
        prefetch_l2(p.g1 + ch * D * D, D * D * 4);
    }
    auto line = [](const void *x) { asm volatile("prefetch.global.L2 [%0];" ::"l"(x)); };
    constexpr int LF = D / 32, LB = D / 64;   // 128-byte lines of a row of floats, of bf16
    for (int e = tid; e < rows * (LF + 3 * LB); e += GT) {
        const int r = e / (LF + 3 * LB), i = e % (LF + 3 * LB);
        const size_t row = ((t0 + r) * p.H + h) * D;
        if (i < LF) line(p.dv + row + 32 * i);
        else {
            const int a = (i - LF) / LB, o = 64 * ((i - LF) % LB);
            line((a == 0 ? p.dout : a == 1 ? p.k : p.q) + row + o);
        }
    }
}

template <int D>
__global__ void __launch_bounds__(GT, 1) kla_bwd_grad_kernel(BwdChunkParams p, int ahead)
{
    constexpr int NB = D / 64, NV = D / 32;       // float4 of half a state per thread
    constexpr int UI = C * D / 8 / GT;            // 8-column items of a [64][D] matrix per thread
    extern __shared__ __align__(128) unsigned char smem_dyn[];
    GradSmem<D> &sm = *reinterpret_cast<GradSmem<D> *>(smem_dyn);
    static_assert(sizeof(GradSmem<D>) <= 232448, "shared memory of one block");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int slot = blockIdx.x / p.H, h = blockIdx.x % p.H;
    const Where w = locate(p, slot);
    if (w.c * C >= w.len) return;
    const int rows = min(C, w.len - w.c * C);
    const size_t t0 = (size_t)w.tok0 + w.c * C, ch = (size_t)slot * p.H + h;
    load_tile<NB, D, GT>(smem_u32(sm.dout), p.dout, t0, rows, p.H, h, 0, tid);
    if (tid < (int)sizeof(Scal) / 16) cp16(smem_u32(&sm.s) + tid * 16, reinterpret_cast<const char *>(p.scal + ch) + tid * 16, true);
    cp_commit();

    // S_0^T / G_1^T, 64 columns of d_k from 64 hh on: tile tt of the 16 rows of d_v from 16 tg on, respectively 8 columns of a row to
    // two float4
    auto tg = [&](int i) { return (warp * NV + i) / 8; };
    auto tt = [&](int i) { return (warp * NV + i) % 8; };
    float4 ps[NV], pg[NV];
    auto fetch = [&](float4 (&pre)[NV], const float *src, int hh) {
        if constexpr (STATE_TILES<D>) {
#pragma unroll
            for (int i = 0; i < NV; ++i) pre[i] = load4(src + ch * D * D + tg(i) * 16 * D + (8 * hh + tt(i)) * 128 + lane * 4);
        } else {
#pragma unroll
            for (int i = 0; i < NV; i += 2) {
                const int e = tid + i / 2 * GT;
                const float *x = src + ch * D * D + (size_t)(e >> 3) * D + hh * 64 + (e & 7) * 8;
                pre[i] = load4(x);
                pre[i + 1] = load4(x + 4);
            }
        }
    };
    auto put8 = [&](unsigned char *dst, int plane, uint32_t off, const float4 &a, const float4 &b) {
        uint32_t hh[4], mm[4], ll[4];
        split3(a.x, a.y, hh[0], mm[0], ll[0]);
        split3(a.z, a.w, hh[1], mm[1], ll[1]);
        split3(b.x, b.y, hh[2], mm[2], ll[2]);
        split3(b.z, b.w, hh[3], mm[3], ll[3]);
        *reinterpret_cast<uint4 *>(dst + off) = make_uint4(hh[0], hh[1], hh[2], hh[3]);
        *reinterpret_cast<uint4 *>(dst + plane + off) = make_uint4(mm[0], mm[1], mm[2], mm[3]);
        *reinterpret_cast<uint4 *>(dst + 2 * plane + off) = make_uint4(ll[0], ll[1], ll[2], ll[3]);
    };
    auto commit = [&](const float4 (&pre)[NV]) {
        if constexpr (STATE_TILES<D>) {
#pragma unroll
            for (int i = 0; i < NV; ++i)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    uint32_t hh, mm, ll;
                    split3(u ? pre[i].z : pre[i].x, u ? pre[i].w : pre[i].y, hh, mm, ll);
                    const uint32_t off = sw128(tg(i) * 16 + u * 8 + (lane >> 2), tt(i)) + 4 * (lane & 3);
                    *reinterpret_cast<uint32_t *>(sm.sg + off) = hh;
                    *reinterpret_cast<uint32_t *>(sm.sg + D * 128 + off) = mm;
                    *reinterpret_cast<uint32_t *>(sm.sg + 2 * D * 128 + off) = ll;
                }
        } else {
#pragma unroll
            for (int i = 0; i < NV; i += 2) {
                const int e = tid + i / 2 * GT;
                put8(sm.sg, D * 128, sw128(e >> 3, e & 7), pre[i], pre[i + 1]);
            }
        }
    };

    // U and lam as operand planes; dbeta_i = (U_i / beta_i) . (lam_i / beta_i)
    {
        float4 a[UI][4];
#pragma unroll
        for (int i = 0; i < UI; ++i) {
            const int e = tid + i * GT, r = e / (D / 8), c8 = e % (D / 8);
            const float *x = p.u + ch * C * D + (size_t)r * D + c8 * 8;
            const float *y = p.dv + ((t0 + (r < rows ? r : 0)) * p.H + h) * D + c8 * 8;
            a[i][0] = load4(x);
            a[i][1] = load4(x + 4);
            a[i][2] = load4(y);
            a[i][3] = load4(y + 4);
        }
        fetch(ps, p.s0, 0);
        if ((int)blockIdx.x + ahead < (int)gridDim.x) prefetch_block<D>(p, blockIdx.x + ahead, tid);
        cp_wait<0>();
        __syncthreads();   // scalars (and dO) are there
#pragma unroll
        for (int i = 0; i < UI; ++i) {
            const int e = tid + i * GT, r = e / (D / 8), c8 = e % (D / 8);
            if (r >= rows) a[i][0] = a[i][1] = a[i][2] = a[i][3] = make_float4(0.f, 0.f, 0.f, 0.f);
            const uint32_t off = (c8 >> 3) * 8192 + sw128(r, c8 & 7);
            put8(sm.u, NB * 8192, off, a[i][0], a[i][1]);
            put8(sm.lam, NB * 8192, off, a[i][2], a[i][3]);
            const float bi = r < rows ? 1.f / sm.s.beta[r] : 0.f;
            float d = (a[i][0].x * bi) * (a[i][2].x * bi) + (a[i][0].y * bi) * (a[i][2].y * bi) + (a[i][0].z * bi) * (a[i][2].z * bi) +
                      (a[i][0].w * bi) * (a[i][2].w * bi) + (a[i][1].x * bi) * (a[i][3].x * bi) + (a[i][1].y * bi) * (a[i][3].y * bi) +
                      (a[i][1].z * bi) * (a[i][3].z * bi) + (a[i][1].w * bi) * (a[i][3].w * bi);
#pragma unroll
            for (int o = D / 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            if (c8 == 0) {
                const float de = p.coeff_eta ? d : d / sm.s.nrm[r];
                if (r < rows) p.deta[(t0 + r) * p.H + h] = de;
                sm.s.dn[r] = p.coeff_eta ? 0.f : -2.f * de * sm.s.beta[r];   // dk_i += this x k_i
            }
        }
    }
    __syncthreads();

    const int r = lane >> 2, cq = 2 * (lane & 3);
    auto ratio = [&](int i, int j) { return exp2f((sm.s.g2h[i] - sm.s.g2h[j]) + (sm.s.g2l[i] - sm.s.g2l[j])); };
    // F = qinv A o (dO U^T) (three terms) and E = -A o (lam U^T) (six), in 16 x 16 blocks on and below the diagonal; their planes hold what
    // lies below it
    auto block = [&](bool is_e, int blk) {
        const int bi = blk < 1 ? 0 : blk < 3 ? 1 : blk < 6 ? 2 : 3, bj = blk - bi * (bi + 1) / 2;
        if (bi * 16 >= rows) return;   // tokens past the end: never read
        float c0[4], c1[4], l0[4], l1[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) c0[e] = c1[e] = l0[e] = l1[e] = 0.f;
        const uint32_t at = smem_u32(is_e ? sm.lam : sm.dout), bt = smem_u32(sm.u);
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {   // the first planes: half of d_v at a time, added in fp32
            float h0[4] = {0.f, 0.f, 0.f, 0.f}, h1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
            for (int kk = 0; kk < D / 32; ++kk) {
                const int ks = half * (D / 32) + kk;
                const uint32_t o = (ks >> 2) * 8192;
                uint32_t a[3][4], b[3][4];
#pragma unroll
                for (int pl = 0; pl < 3; ++pl) frag_b(b[pl], bt + pl * NB * 8192 + o, (ks & 3) * 16, bj * 16, lane);
                frag_a(a[0], at + o, bi * 16, (ks & 3) * 16, lane);
                mma(h0, a[0], b[0][0], b[0][1]);
                mma(h1, a[0], b[0][2], b[0][3]);
                if (is_e) {
                    frag_a(a[1], at + NB * 8192 + o, bi * 16, (ks & 3) * 16, lane);
                    frag_a(a[2], at + 2 * NB * 8192 + o, bi * 16, (ks & 3) * 16, lane);
                    mma5(l0, l1, a, b);
                } else {
#pragma unroll
                    for (int pl = 2; pl > 0; --pl) {
                        mma(l0, a[0], b[pl][0], b[pl][1]);
                        mma(l1, a[0], b[pl][2], b[pl][3]);
                    }
                }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) c0[e] += h0[e], c1[e] += h1[e];
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) c0[e] += l0[e], c1[e] += l1[e];
        unsigned char *dst = is_e ? sm.e : sm.f;
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                const int i = bi * 16 + r + (e >> 1) * 8, j = bj * 16 + t * 8 + cq;
                const float sc = is_e ? -1.f : sm.s.qinv[i];
                float x = t ? c1[e] : c0[e], y = t ? c1[e + 1] : c0[e + 1];
                if (!is_e && j == (i & ~1)) sm.s.beta[i] = sc * (j == i ? x : y);   // the diagonal of F (the betas have been used)
                x = j < i ? sc * ratio(i, j) * x : 0.f;
                y = j + 1 < i ? sc * ratio(i, j + 1) * y : 0.f;
                uint32_t hh, mm, ll;
                split3(x, y, hh, mm, ll);
                const uint32_t off = sw128(i, bj * 2 + t) + 4 * (lane & 3);
                *reinterpret_cast<uint32_t *>(dst + off) = hh;
                *reinterpret_cast<uint32_t *>(dst + 8192 + off) = mm;
                *reinterpret_cast<uint32_t *>(dst + 16384 + off) = ll;
            }
    };
    // ten blocks of each, an E block costs two F blocks
    if (warp < 10) block(true, warp);
    else
        for (int b = warp - 10; b < 10; b += 6) block(false, b);

    const int mt = warp & 3, nh = warp >> 2, i0 = mt * 16;   // this warp's 16 tokens and 16 of the half's 64 columns
    const int ia = i0 + r, ib = ia + 8;
    const int ks_s = i0 < rows ? D / 16 : 0;      // a warp whose tokens all lie past the end takes no part in the products
    const int ks_j = (rows + 15) / 16;            // token blocks that hold any
    float gs = 0.f;             // this thread's part of gC <G_1, S_0>
    float dga = 0.f, dgb = 0.f; // ... of dg of its two rows, without
    float cja = 0.f, cjb = 0.f; // ... what they have in common with <G_1, S_1>
    const float gama = sm.s.gam[ia], gamb = sm.s.gam[ib], deca = sm.s.dec[ia], decb = sm.s.dec[ib], gc = sm.s.gam[C - 1];
    const float qia = sm.s.qinv[ia], qib = sm.s.qinv[ib];
    auto pair = [&](const unsigned char *tile, int i, int t) { return unpack(*reinterpret_cast<const uint32_t *>(tile + sw128(i, nh * 2 + t) + 4 * (lane & 3))); };
    // products x . y of this lane's elements of the two rows, added to a and b
    auto dot = [&](const unsigned char *tile, const float (&x)[2][4], float &a, float &b) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const float2 fa = pair(tile, ia, t), fb = pair(tile, ib, t);
            a += fa.x * x[t][0] + fa.y * x[t][1];
            b += fb.x * x[t][2] + fb.y * x[t][3];
        }
    };
    const uint32_t sg = smem_u32(sm.sg), kt = smem_u32(sm.k), qt = smem_u32(sm.q);
#pragma unroll 1
    for (int hh = 0; hh < NB; ++hh) {
        load_tile<1, D, GT>(kt, p.k, t0, rows, p.H, h, hh * 64, tid);
        load_tile<1, D, GT>(qt, p.q, t0, rows, p.H, h, hh * 64, tid);
        cp_commit();
        commit(ps);
        fetch(pg, p.g1, hh);
        cp_wait<0>();
        __syncthreads();   // S_0 planes, K, Q (and, the first time, E and F)
        float xq[2][4], xk[2][4], yq[2][4], yk[2][4];   // y: the lower planes' part
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) xq[t][e] = xk[t][e] = yq[t][e] = yk[t][e] = 0.f;
        // dO S_0^T and lam S_0^T
#pragma unroll 2
        for (int ks = 0; ks < ks_s; ++ks) {
            const uint32_t o = (ks >> 2) * 8192;
            uint32_t a[4], l[3][4], b[3][4];
            frag_a(a, smem_u32(sm.dout) + o, i0, (ks & 3) * 16, lane);
#pragma unroll
            for (int pl = 0; pl < 3; ++pl) frag_a(l[pl], smem_u32(sm.lam) + pl * NB * 8192 + o, i0, (ks & 3) * 16, lane);
#pragma unroll
            for (int pl = 0; pl < 3; ++pl) frag_bt(b[pl], sg + pl * D * 128, ks * 16, nh * 16, lane);
            mma(xq[0], a, b[0][0], b[0][1]);
            mma(xq[1], a, b[0][2], b[0][3]);
            mma(xk[0], l[0], b[0][0], b[0][1]);
            mma(xk[1], l[0], b[0][2], b[0][3]);
#pragma unroll
            for (int pl = 2; pl > 0; --pl) {
                mma(yq[0], a, b[pl][0], b[pl][1]);
                mma(yq[1], a, b[pl][2], b[pl][3]);
            }
            mma5(yk[0], yk[1], l, b);
        }
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                xq[t][e] += yq[t][e];
                xk[t][e] += yk[t][e];
                yq[t][e] = yk[t][e] = 0.f;
            }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            xq[t][0] *= gama * qia; xq[t][1] *= gama * qia; xq[t][2] *= gamb * qib; xq[t][3] *= gamb * qib;
            xk[t][0] *= -gama; xk[t][1] *= -gama; xk[t][2] *= -gamb; xk[t][3] *= -gamb;
        }
        // += F K and E K
#pragma unroll 1
        for (int ks = 0; ks <= mt && mt < ks_j; ++ks) {
            uint32_t a[3][4], l[3][4], b[4];
            float hq[2][4], hk[2][4];
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) hq[t][e] = hk[t][e] = 0.f;
#pragma unroll
            for (int pl = 0; pl < 3; ++pl) {
                frag_a(a[pl], smem_u32(sm.f) + pl * 8192, i0, ks * 16, lane);
                frag_a(l[pl], smem_u32(sm.e) + pl * 8192, i0, ks * 16, lane);
            }
            frag_bt(b, kt, ks * 16, nh * 16, lane);
            mma(hq[0], a[0], b[0], b[1]);
            mma(hq[1], a[0], b[2], b[3]);
            mma(hk[0], l[0], b[0], b[1]);
            mma(hk[1], l[0], b[2], b[3]);
#pragma unroll
            for (int pl = 2; pl > 0; --pl) {
                mma(yq[0], a[pl], b[0], b[1]);
                mma(yq[1], a[pl], b[2], b[3]);
                mma(yk[0], l[pl], b[0], b[1]);
                mma(yk[1], l[pl], b[2], b[3]);
            }
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    xq[t][e] += hq[t][e];
                    xk[t][e] += hk[t][e];
                }
        }
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                xq[t][e] += yq[t][e];
                xk[t][e] += yk[t][e];
            }
        // dg from dq and dk without the diagonal of F: no decay acts on it, and its shares of q . dq and k . dk, which under strong decay
        // are nearly all of both, would have to cancel
        dot(sm.q, xq, dga, dgb);
        dot(sm.k, xk, dga, dgb);
        // dq (with the normalised read-out its projection follows below)
        const float fda = sm.s.beta[ia], fdb = sm.s.beta[ib];
        const size_t ga = ((t0 + ia) * p.H + h) * D + hh * 64 + nh * 16 + cq, gb = ga + (size_t)8 * p.H * D;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const float2 ka = pair(sm.k, ia, t), kb = pair(sm.k, ib, t);
            if (ia < rows) store2(p.dq + ga + 8 * t, xq[t][0] + fda * ka.x, xq[t][1] + fda * ka.y);
            if (ib < rows) store2(p.dq + gb + 8 * t, xq[t][2] + fdb * kb.x, xq[t][3] + fdb * kb.y);
        }
        __syncthreads();   // the S_0 planes have been read
#pragma unroll
        for (int i = 0; i < NV; ++i) gs += gc * (ps[i].x * pg[i].x + ps[i].y * pg[i].y + ps[i].z * pg[i].z + ps[i].w * pg[i].w);
        commit(pg);
        if (hh + 1 < NB) fetch(ps, p.s0, hh + 1);
        __syncthreads();
        // D U G_1^T
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) xq[t][e] = yq[t][e] = 0.f;
#pragma unroll 2
        for (int ks = 0; ks < ks_s; ++ks) {
            uint32_t a[3][4], b[3][4];
#pragma unroll
            for (int pl = 0; pl < 3; ++pl) frag_a(a[pl], smem_u32(sm.u) + (pl * NB + (ks >> 2)) * 8192, i0, (ks & 3) * 16, lane);
#pragma unroll
            for (int pl = 0; pl < 3; ++pl) frag_bt(b[pl], sg + pl * D * 128, ks * 16, nh * 16, lane);
            mma(xq[0], a[0], b[0][0], b[0][1]);
            mma(xq[1], a[0], b[0][2], b[0][3]);
            mma5(yq[0], yq[1], a, b);
        }
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) xq[t][e] += yq[t][e];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            xq[t][0] *= deca; xq[t][1] *= deca; xq[t][2] *= decb; xq[t][3] *= decb;
        }
        dot(sm.k, xq, cja, cjb);   // <G_1, S_1> = gC <G_1, S_0> + sum_j k_j . (D U G_1^T)_j
        // += E^T K + F^T Q: rows of this warp are the columns of E and F
        {
            float y[2][4], z[2][4];
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) y[t][e] = z[t][e] = 0.f;
#pragma unroll 1
            for (int ks = mt; ks < ks_j; ++ks) {
                uint32_t a[3][4], l[3][4], b[4], b2[4];
                float h[2][4];
#pragma unroll
                for (int e = 0; e < 4; ++e) h[0][e] = h[1][e] = 0.f;
#pragma unroll
                for (int pl = 0; pl < 3; ++pl) {
                    frag_at(a[pl], smem_u32(sm.f) + pl * 8192, i0, ks * 16, lane);
                    frag_at(l[pl], smem_u32(sm.e) + pl * 8192, i0, ks * 16, lane);
                }
                frag_bt(b, qt, ks * 16, nh * 16, lane);
                frag_bt(b2, kt, ks * 16, nh * 16, lane);
                mma(h[0], a[0], b[0], b[1]);
                mma(h[1], a[0], b[2], b[3]);
                mma(h[0], l[0], b2[0], b2[1]);
                mma(h[1], l[0], b2[2], b2[3]);
#pragma unroll
                for (int pl = 2; pl > 0; --pl) {
                    mma(y[0], a[pl], b[0], b[1]);
                    mma(y[1], a[pl], b[2], b[3]);
                    mma(y[0], l[pl], b2[0], b2[1]);
                    mma(y[1], l[pl], b2[2], b2[3]);
                }
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int e = 0; e < 4; ++e) z[t][e] += h[t][e];
            }
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) z[t][e] += y[t][e];
            float ca = 0.f, cb = 0.f;
            dot(sm.k, z, ca, cb);
            dga -= ca;
            dgb -= cb;
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) xq[t][e] += z[t][e];
        }
        const float na = sm.s.dn[ia], nb = sm.s.dn[ib];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const float2 ka = pair(sm.k, ia, t), kb = pair(sm.k, ib, t), qa = pair(sm.q, ia, t), qb = pair(sm.q, ib, t);
            if (ia < rows) store2(p.dk + ga + 8 * t, (xk[t][0] + xq[t][0]) + (na * ka.x + fda * qa.x), (xk[t][1] + xq[t][1]) + (na * ka.y + fda * qa.y));
            if (ib < rows) store2(p.dk + gb + 8 * t, (xk[t][2] + xq[t][2]) + (nb * kb.x + fdb * qb.x), (xk[t][3] + xq[t][3]) + (nb * kb.y + fdb * qb.y));
        }
        __syncthreads();   // K, Q and the planes may be overwritten
    }

    // dlog_alpha_t = <G_1, S_1> + sum_{i >= t} dg_i; the write of token j is in the first with c_j = k_j . (D U G_1^T)_j and in dg_j with -c_j,
    // the same fp32 value, so that what no decay has touched cancels exactly
    float (*cj)[64] = reinterpret_cast<float (*)[64]>(sm.f);   // (F has been used)
    auto quad = [](float x) {
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        return x + __shfl_xor_sync(0xffffffffu, x, 2);
    };
    dga = quad(dga);
    dgb = quad(dgb);
    cja = quad(cja);
    cjb = quad(cjb);
    if ((lane & 3) == 0) {
        sm.red[nh][ia] = dga;
        sm.red[nh][ib] = dgb;
        cj[nh][ia] = cja;
        cj[nh][ib] = cjb;
    }
    gs = warp_sum(gs);
    if (lane == 0) sm.s.nrm[warp] = gs;   // (the norms have been used; no room for an array of its own at d = 128)
    __syncthreads();
    if (warp == 0) {
        double tot = 0.0;
#pragma unroll
        for (int i = 0; i < GW; ++i) tot += (double)sm.s.nrm[i];
        auto rsum = [](const float (*r)[64], int i) { return ((double)r[0][i] + (double)r[1][i]) + ((double)r[2][i] + (double)r[3][i]); };
        const int a = 63 - 2 * lane, b = a - 1;   // lane 0 holds the last two tokens
        const double c0 = rsum(cj, a), c1 = rsum(cj, b);
        double c = c0 + c1;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        tot += c;
        const double x0 = rsum(sm.red, a) - c0, x1 = rsum(sm.red, b) - c1;
        double incl = x0 + x1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (a < rows) p.dlog_alpha[(t0 + a) * p.H + h] = (float)(tot + incl - x1);
        if (b < rows) p.dlog_alpha[(t0 + b) * p.H + h] = (float)(tot + incl);
    } else if (p.qnorm) {
        // z = dq so far; q^ = q / ||q||: dq = z - q^ (q^ . z), the read-out's projection (the block's own stores, after the barrier)
        for (int i = warp - 1; i < rows; i += GW - 1) {
            const size_t g = ((t0 + i) * p.H + h) * D;
            float z[D / 32], q[D / 32], s = 0.f;
#pragma unroll
            for (int j = 0; j < D / 32; ++j) {
                z[j] = p.dq[g + lane + 32 * j];
                q[j] = to_f32(p.q[g + lane + 32 * j]) * sm.s.qinv[i];
                s += q[j] * z[j];
            }
            s = warp_sum(s);
#pragma unroll
            for (int j = 0; j < D / 32; ++j) p.dq[g + lane + 32 * j] = z[j] - q[j] * s;
        }
    }
}

// ---- host side ------------------------------------------------------------------------------------------------------------
template <typename K>
cudaError_t allow_smem(K kern, int bytes)
{
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

template <int D>
cudaError_t launch_d(const BwdChunkParams &p, uint64_t n_tok, cudaStream_t stream)
{
    const int smem1 = (int)sizeof(PrepSmem<D>), smem2 = (int)sizeof(ChainSmem<D>), smem3 = (int)sizeof(GradSmem<D>);
    cudaError_t e = allow_smem(kla_bwd_prepare_kernel<D>, smem1);
    if (e == cudaSuccess) e = allow_smem(kla_bwd_chain_kernel<D>, smem2);
    if (e == cudaSuccess) e = allow_smem(kla_bwd_grad_kernel<D>, smem3);
    if (e != cudaSuccess) return e;
    const int units = p.n_seq * p.H * (D / 64);
    if (units == 0) return cudaSuccess;
    TileMaps tm = {};
    const uint64_t row = (uint64_t)p.H * D;
    if (n_tok > 0 && (!make_tile_map(&tm.q, p.q, n_tok, row) || !make_tile_map(&tm.k, p.k, n_tok, row) ||
                      !make_tile_map(&tm.v, p.v, n_tok, row) || !make_tile_map(&tm.dout, p.dout, n_tok, row)))
        return cudaErrorInvalidValue;
    if (p.n_slots > 0) kla_bwd_prepare_kernel<D><<<p.n_slots * p.H, 256, smem1, stream>>>(p);
    kla_bwd_chain_kernel<D><<<2 * units, 128, smem2, stream>>>(tm, p, units);   // (empty sequences: dinit)
    if (p.n_slots > 0) kla_bwd_grad_kernel<D><<<p.n_slots * p.H, GT, smem3, stream>>>(p, sm_count());
    count_launch(p.n_slots > 0 ? 3 : 1);
    return cudaGetLastError();
}

// Bytes of the workspace areas of one (slot, head), each a multiple of 1024.
constexpr size_t per_entry(int d) { return (size_t)T_BYTES + 2 * (size_t)d * C * 4 + 2 * (size_t)d * d * 4 + sizeof(Scal); }
size_t order_area(int n_seq) { return ((size_t)n_seq * 4 + 1023) & ~(size_t)1023; }

}  // namespace

size_t bwd_chunk_workspace_bytes(int n_seq, long long n_tok, int H, int d)
{
    return order_area(n_seq) + (size_t)(n_tok / C + n_seq) * H * per_entry(d);
}

cudaError_t launch_bwd_chunk(const BwdArgs &a, cudaStream_t stream)
{
    BwdChunkParams p;
    p.q = (const __nv_bfloat16 *)a.q; p.k = (const __nv_bfloat16 *)a.k; p.v = (const __nv_bfloat16 *)a.v; p.dout = (const __nv_bfloat16 *)a.dout;
    p.log_alpha = a.log_alpha; p.eta = a.eta;
    p.init_state = a.init_state; p.dfinal = a.dfinal;
    p.dq = a.dq; p.dk = a.dk; p.dv = a.dv; p.dlog_alpha = a.dlog_alpha; p.deta = a.deta; p.dinit = a.dinit;
    p.cu_seqlens = a.cu_seqlens;
    p.T = a.T; p.H = a.H; p.n_seq = a.n_seq;
    p.eps = a.eps;
    p.coeff_eta = a.coeff_eta; p.qnorm = a.qnorm;
    p.n_slots = a.cu_seqlens ? (int)(a.n_tok / C) + a.n_seq : a.n_seq * ((a.T + C - 1) / C);
    p.order = nullptr;
    // longest first only where the chains' blocks do not all start at once (the order takes quadratic work)
    if (a.cu_seqlens && a.n_seq > 1 && a.n_seq <= 4096 && 2LL * a.n_seq * a.H * (a.d / 64) > sm_count()) {
        int32_t *order = (int32_t *)a.workspace;
        const cudaError_t e = launch_seq_order(a.cu_seqlens, a.n_seq, order, stream);
        if (e != cudaSuccess) return e;
        p.order = order;
    }
    const size_t n = (size_t)p.n_slots * a.H, d = (size_t)a.d;
    unsigned char *w = (unsigned char *)a.workspace + order_area(a.n_seq);
    p.tpl = w;
    w += n * T_BYTES;
    p.pdo = (float *)w;
    w += n * d * C * 4;
    p.u = (float *)w;
    w += n * d * C * 4;
    p.s0 = (float *)w;
    w += n * d * d * 4;
    p.g1 = (float *)w;
    w += n * d * d * 4;
    p.scal = (Scal *)w;
    p.test_timeout = a.test_timeout;
    p.status_word = a.status_word;
    return a.d == 128 ? launch_d<128>(p, (uint64_t)a.n_tok, stream) : launch_d<64>(p, (uint64_t)a.n_tok, stream);
}

}  // namespace kla
