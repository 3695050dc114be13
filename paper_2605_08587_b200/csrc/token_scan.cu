// The recurrence on CUDA cores in fp32, four tokens at a time (Algorithm 1, left panel; Appendix B.5 for diagonal gates).
//
//     S~ = diag(alpha_t) S_{t-1},   e_t = v_t - S~^T k_t,   beta_t = eta_t / (||k_t||^2 + eps)   (Eq. 3)
//     S_t = S~ + beta_t k_t e_t^T,  o_t = S_t^T q_t
//
// with alpha_t one number (chunk forward on fp32 inputs or with chunk 16 / 32) or one
// number per row of the state (diagonal gates).  The result does not depend on a chunk length, so none is used.
//
// Four tokens of a head form a block; with A_t the product of the decays up to token t of the block,
//
//     u_t = S_0^T (A_t o k_t),  w_t = S_0^T (A_t o q_t)                          one sweep over the state for all four
//     e_t = v_t - u_t - sum_{s<t} Lk_ts e_s,   o_t = w_t + sum_{s<=t} Lq_ts e_s   4 x 4 triangles
//     S_4 = A_4 o S_0 + sum_s (beta_s k_s o A_4/A_s) e_s                          one update of the state for all four
//
// where Lk_ts = beta_s k_t . (A_t/A_s o k_s) and Lq likewise with q_t.  All decay ratios are products of alphas (never a
// quotient), so nothing overflows however strong the decay.  A_4 itself, which the state meets with every block, is applied with its
// rounding error (expm1 of the sum of log alpha where it is near 1): an error of 2^-25 in a decay near 1 is the same for the whole
// state and, of one sign as those of expf are, adds up over all that is remembered (log alpha / 100, eta / 10, 4 096 tokens, fp32: final
// state off by 5.9e-6 of its norm with A_4 as a product of four expf, 4.7e-7 this way).  What depends on the head only -- the decayed
// vectors, the triangles, beta -- is prepared once per block of tokens by one warp and read by every warp from shared memory.
//
// What bounds it: the fp32 pipe.  A token costs 3.5 d^2 multiply-adds per head (2 d^2 in the sweep, d^2 in the update, half
// for the decay and its rounding error), fewer than the chunk algebra on the same cores (4 C d + 6 d^2 flops, half as multiply-adds, plus
// the triangular solve), and the four-token block divides the latency of the reductions by four (one token at a time, the
// scan of a layer with diagonal gates, B8 H8 T4096 d128, took 2.94 ms: 1 370 cycles per token for 340 cycles of arithmetic; the
// chunk algebra on CUDA cores took 102 us for the 256 tokens of the small fp32 configuration, this scan 33 us).
// Columns of the state never interact (the write is k e^T), so a warp owns 4 CPL of them for the whole sequence and no
// scanning warp talks to another; as many warps beside them prepare the next blocks, so that their work fills the issue slots
// the multiply-adds leave.  Lane = (row group rg = lane & 7, CPL columns at lane >> 3): rows 4 (rg + 8 i) .. + 3 of these
// columns, in registers.  That layout reads every operand as float4 without bank conflicts, pairs adjacent rows into packed
// fp32 multiply-adds without duplicating an operand, and leaves only three butterfly stages for the sums over rows.
// CPL: a float4 from shared memory costs four cycles of the load pipe even when it is a broadcast, and feeds 2 CPL packed
// multiply-adds (four SM cycles at CPL = 4): with CPL = 2 the scan of a layer was bound by those loads (1.40 ms; with
// CPL = 4 and both sweeps in one loop 1.00 ms, 1.06 with the decay's rounding error, bound by the latency of one scanning warp per
// scheduler: fp32 pipe 56 % busy, load pipe 25 %, schedulers 50 %).  CPL = 2 stays where there are too few (sequence, head) pairs to give every SM more than
// two warps of 16 columns: twice the warps then halve the latency.
#include "common.cuh"
#include "scan_pieces.cuh"

namespace kla {

namespace {

constexpr int BT = 4;     // tokens per block
constexpr int NW = 4;     // scanning warps per thread block, and as many preparing ones: one of each per scheduler

// One block of BT tokens as the scan reads it.
template <int D, int CPL, bool DIAG>
struct Block {
    float k[BT][D], q[BT][D];    // A_t o k_t, A_t o q_t
    float b[BT][D];              // beta_s k_s o A_4 / A_s
    float decay[DIAG ? D : 4];      // A_4 rounded (without diagonal gates one number, [0])
    float decay_lo[DIAG ? D : 4];   // what the rounding left out
    float tri[BT][BT];           // [t][s], s <= t: Lq_ts;  [s][t], s < t: Lk_ts
    float v[BT][NW * 4 * CPL];   // the thread block's columns
};

template <int D, int CPL, typename IO, typename OUT, bool DIAG>
__global__ void __launch_bounds__(64 * NW, 1) kla_token_scan_kernel(TokenScanParams p)
{
    using Blk = Block<D, CPL, DIAG>;
    constexpr int WCOLS = 4 * CPL, COLS = NW * WCOLS, GROUPS = D / COLS;   // columns per warp, per thread block
    constexpr int VL = CPL / 2;                                            // sums per lane after the butterflies
    constexpr int VC = COLS / 8;                                           // columns of v per lane in the preparation
    constexpr int NI = D / 32;   // float4 row groups per lane
    constexpr int JD = D / 32;   // state rows per lane in the preparation
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Blk *const stage = reinterpret_cast<Blk *>(smem_raw);   // two stages of NW blocks
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rg = lane & 7, cp = lane >> 3;
    const int cg = blockIdx.x % GROUPS, h = (blockIdx.x / GROUPS) % p.H, n = blockIdx.x / (GROUPS * p.H);
    int len;
    int tok0;
    if (p.cu_seqlens) {
        tok0 = p.cu_seqlens[n];
        len = p.cu_seqlens[n + 1] - tok0;
    } else {
        tok0 = n * p.T;
        len = p.T;
    }
    const size_t row0 = (size_t)tok0 * p.H + h, stride = (size_t)p.H;   // token t of this (sequence, head) is row row0 + t * stride
    const IO *qp = reinterpret_cast<const IO *>(p.q), *kp = reinterpret_cast<const IO *>(p.k), *vp = reinterpret_cast<const IO *>(p.v);
    OUT *op = reinterpret_cast<OUT *>(p.out);

    // ---- preparation: one warp per block of tokens, lane l holds rows l JD .. + JD - 1 ------------------------------------
    struct Raw {
        IO k[BT][JD], q[BT][JD];
        Vec4<IO> v[VC / 4];            // VC columns of token lane / 8
        float la[DIAG ? BT : 1][DIAG ? JD : 1];
        float la_s, eta;               // scalar gate and eta of token lane & 3
    };
    auto load_j = [&](IO (&dst)[JD], const IO *src) {
        if constexpr (sizeof(IO) * JD == 16) *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(src);
        else if constexpr (sizeof(IO) * JD == 8) *reinterpret_cast<uint2 *>(dst) = *reinterpret_cast<const uint2 *>(src);
        else *reinterpret_cast<uint32_t *>(dst) = *reinterpret_cast<const uint32_t *>(src);
    };
    auto request = [&](Raw &r, int t0) {
#pragma unroll
        for (int t = 0; t < BT; ++t) {
            const size_t row = row0 + (size_t)min(t0 + t, len - 1) * stride;
            load_j(r.k[t], kp + row * D + lane * JD);
            load_j(r.q[t], qp + row * D + lane * JD);
            if constexpr (DIAG) {
                if constexpr (JD == 4) *reinterpret_cast<float4 *>(r.la[t]) = *reinterpret_cast<const float4 *>(p.log_alpha + row * D + lane * JD);
                else *reinterpret_cast<float2 *>(r.la[t]) = *reinterpret_cast<const float2 *>(p.log_alpha + row * D + lane * JD);
            }
        }
        const size_t row = row0 + (size_t)min(t0 + (lane & 3), len - 1) * stride;
        if constexpr (!DIAG) r.la_s = p.log_alpha[row];
        r.eta = p.eta[row];
        const IO *src = vp + (row0 + (size_t)min(t0 + cp, len - 1) * stride) * D + cg * COLS + rg * VC;
#pragma unroll
        for (int i = 0; i < VC; i += 4) r.v[i / 4].load(src + i);
    };
    auto commit = [&](Blk &bl, const Raw &r, int t0) {
        float k[BT][JD], q[BT][JD], a[BT][JD];
        float nk[BT], nq[BT];
#pragma unroll
        for (int t = 0; t < BT; ++t) {
            const bool in = t0 + t < len;   // tokens past the end: k = q = 0, alpha = 1, beta = 0
            const float as = DIAG ? 1.f : expf(__shfl_sync(0xffffffffu, r.la_s, t));
            nk[t] = nq[t] = 0.f;
#pragma unroll
            for (int j = 0; j < JD; ++j) {
                k[t][j] = in ? to_f32(r.k[t][j]) : 0.f;
                q[t][j] = in ? to_f32(r.q[t][j]) : 0.f;
                if constexpr (DIAG) a[t][j] = in ? expf(r.la[t][j]) : 1.f;
                else a[t][j] = in ? as : 1.f;
                nk[t] += k[t][j] * k[t][j];
                nq[t] += q[t][j] * q[t][j];
            }
        }
        const float nrm = reduce_scatter<4>(nk, lane);   // of token (lane >> 3) & 3
        const float eta = __shfl_sync(0xffffffffu, r.eta, cp);
        const float beta_mine = t0 + cp < len ? (p.coeff_eta ? eta : eta / (nrm + p.eps)) : 0.f;   // Eq. 3
        float beta[BT];
#pragma unroll
        for (int t = 0; t < BT; ++t) beta[t] = __shfl_sync(0xffffffffu, beta_mine, lane_of_col<4>(t));
        if (p.qnorm) {   // read-out over ||q||
            const float qi = reduce_scatter<4>(nq, lane);
#pragma unroll
            for (int t = 0; t < BT; ++t) {
                const float x = t0 + t < len ? 1.f / sqrtf(__shfl_sync(0xffffffffu, qi, lane_of_col<4>(t))) : 0.f;
#pragma unroll
                for (int j = 0; j < JD; ++j) q[t][j] *= x;
            }
        }
        // triangles: x[row * 4 + col] = Lq[row][col] (col <= row) or Lk[col][row] (col > row), without the factor beta
        float x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = 0.f;
#pragma unroll
        for (int j = 0; j < JD; ++j) {
#pragma unroll
            for (int s = 0; s < BT; ++s) {
                float ks = k[s][j];
                x[s * 4 + s] += q[s][j] * ks;
#pragma unroll
                for (int t = s + 1; t < BT; ++t) {
                    ks *= a[t][j];
                    x[t * 4 + s] += q[t][j] * ks;
                    x[s * 4 + t] += k[t][j] * ks;
                }
            }
        }
#pragma unroll
        for (int n2 = 16, off = 16; n2 > 1; n2 >>= 1, off >>= 1) {
            const bool hi = lane & off;
#pragma unroll
            for (int i = 0; i < n2 / 2; ++i) {
                const float keep = hi ? x[n2 / 2 + i] : x[i], give = hi ? x[i] : x[n2 / 2 + i];
                x[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
            }
        }
        const float tri = x[0] + __shfl_xor_sync(0xffffffffu, x[0], 1);
        const int tr = lane >> 3, tc = (lane >> 1) & 3;   // the sum this lane ended up with
        if ((lane & 1) == 0) {
            const int s = min(tr, tc);
            const float bs = s == 0 ? beta[0] : s == 1 ? beta[1] : s == 2 ? beta[2] : beta[3];
            bl.tri[tr][tc] = bs * tri;
        }
        auto put = [&](float *dst, const float (&y)[JD]) {
            if constexpr (JD == 4) *reinterpret_cast<float4 *>(dst + lane * 4) = make_float4(y[0], y[1], y[2], y[3]);
            else *reinterpret_cast<float2 *>(dst + lane * 2) = make_float2(y[0], y[1]);
        };
        float A[JD];
#pragma unroll
        for (int j = 0; j < JD; ++j) A[j] = 1.f;
#pragma unroll
        for (int t = 0; t < BT; ++t) {
            float y[JD], z[JD];
#pragma unroll
            for (int j = 0; j < JD; ++j) {
                A[j] *= a[t][j];
                y[j] = A[j] * k[t][j];
                z[j] = A[j] * q[t][j];
            }
            put(bl.k[t], y);
            put(bl.q[t], z);
        }
        float lo[JD];
#pragma unroll
        for (int j = 0; j < JD; ++j) {
            float sum = 0.f;
#pragma unroll
            for (int t = 0; t < BT; ++t) {
                const float la = DIAG ? r.la[DIAG ? t : 0][DIAG ? j : 0] : __shfl_sync(0xffffffffu, r.la_s, t);
                sum += t0 + t < len ? la : 0.f;
            }
            const float m = expm1f(sum), hi = 1.f + m;
            lo[j] = A[j] > 0.5f ? (1.f - hi) + m : 0.f;
            if (A[j] > 0.5f) A[j] = hi;
            if (!DIAG) break;   // one number for all rows
        }
        if constexpr (DIAG) {
            put(bl.decay, A);
            put(bl.decay_lo, lo);
        } else if (lane == 0) {
            bl.decay[0] = A[0];
            bl.decay_lo[0] = lo[0];
        }
#pragma unroll
        for (int j = 0; j < JD; ++j) A[j] = 1.f;
#pragma unroll
        for (int t = BT - 1; t >= 0; --t) {
            float y[JD];
#pragma unroll
            for (int j = 0; j < JD; ++j) {
                y[j] = beta[t] * k[t][j] * A[j];
                A[j] *= a[t][j];
            }
            put(bl.b[t], y);
        }
#pragma unroll
        for (int i = 0; i < VC; i += 4) store4(&bl.v[cp][rg * VC + i], r.v[i / 4].get());
    };

    // stage s holds the tokens s NW BT .. of the sequence, block m of it at stage[(s & 1) NW + m]
    const int nst = (len + NW * BT - 1) / (NW * BT);
    if (warp >= NW) {
        // ---- preparing warps: block `mine` of every stage, one stage ahead of the scan, requested two ahead ----------------
        const int mine = warp - NW;
        Raw raw;
        auto first = [&](int st) { return (st * NW + mine) * BT; };
        if (len > 0) request(raw, first(0));
        for (int st = 0; st <= nst; ++st) {   // in iteration st the scan works on stage st - 1
            if (st < nst) {
                if (first(st) < len) commit(stage[(st & 1) * NW + mine], raw, first(st));
                if (st + 1 < nst) request(raw, first(st + 1));
            }
            __syncthreads();
        }
        return;
    }

    // ---- scanning warps --------------------------------------------------------------------------------------------------
    const int c0 = cg * COLS + warp * WCOLS + cp * CPL;   // this lane's CPL columns
    const size_t sbase = ((size_t)n * p.H + h) * D * D + c0;
    // S[i][u][c] = rows (4 (rg + 8 i) + 2 u, + 1) of column c0 + c
    float2 S[NI][2][CPL];
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < CPL; c += 2) {
                float2 x = f2(0.f);
                if (p.init_state) x = *reinterpret_cast<const float2 *>(p.init_state + sbase + (size_t)(4 * (rg + 8 * i) + r) * D + c);
                if (r & 1) {
                    S[i][r >> 1][c].y = x.x;
                    S[i][r >> 1][c + 1].y = x.y;
                } else {
                    S[i][r >> 1][c].x = x.x;
                    S[i][r >> 1][c + 1].x = x.y;
                }
            }

    auto process = [&](const Blk &bl, int t0) {
        const float d0 = bl.decay[0], d1 = bl.decay_lo[0];
        // one sweep over the state for k and q of all four tokens
        float2 au[BT][CPL], aw[BT][CPL];
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
            for (int t = 0; t < BT; ++t) {
                const float4 x = load4(&bl.k[t][4 * (rg + 8 * i)]), y = load4(&bl.q[t][4 * (rg + 8 * i)]);
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    au[t][c] = i == 0 ? mul2(f2(x.x, x.y), S[i][0][c]) : fma2(f2(x.x, x.y), S[i][0][c], au[t][c]);
                    aw[t][c] = i == 0 ? mul2(f2(y.x, y.y), S[i][0][c]) : fma2(f2(y.x, y.y), S[i][0][c], aw[t][c]);
                }
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    au[t][c] = fma2(f2(x.z, x.w), S[i][1][c], au[t][c]);
                    aw[t][c] = fma2(f2(y.z, y.w), S[i][1][c], aw[t][c]);
                }
            }
        // sums over the eight row groups: this lane ends up with token rg >> 1, columns (rg & 1) VL .. + VL - 1 of its CPL
        float yu[BT * CPL], yw[BT * CPL];
#pragma unroll
        for (int t = 0; t < BT; ++t)
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                yu[t * CPL + c] = au[t][c].x + au[t][c].y;
                yw[t * CPL + c] = aw[t][c].x + aw[t][c].y;
            }
#pragma unroll
        for (int n2 = BT * CPL, off = 4; off > 0; n2 >>= 1, off >>= 1) {
            const bool hi = lane & off;
#pragma unroll
            for (int i = 0; i < n2 / 2; ++i) {
                const float keep = hi ? yu[n2 / 2 + i] : yu[i], give = hi ? yu[i] : yu[n2 / 2 + i];
                yu[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
            }
#pragma unroll
            for (int i = 0; i < n2 / 2; ++i) {
                const float keep = hi ? yw[n2 / 2 + i] : yw[i], give = hi ? yw[i] : yw[n2 / 2 + i];
                yw[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
            }
        }
        float u[VL], w[VL];
#pragma unroll
        for (int x = 0; x < VL; ++x) {
            u[x] = yu[x];
            w[x] = yw[x];
        }
        float tri[BT][BT];
#pragma unroll
        for (int t = 0; t < BT; ++t) *reinterpret_cast<float4 *>(tri[t]) = load4(bl.tri[t]);
        float e[BT][CPL];
#pragma unroll
        for (int t = 0; t < BT; ++t) {
            float v[CPL];
#pragma unroll
            for (int c = 0; c < CPL; c += 2)
                *reinterpret_cast<float2 *>(&v[c]) = *reinterpret_cast<const float2 *>(&bl.v[t][warp * WCOLS + cp * CPL + c]);
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                float x = v[c] - __shfl_sync(0xffffffffu, u[c % VL], (lane & 24) | (2 * t + c / VL));
#pragma unroll
                for (int s = 0; s < t; ++s) x -= tri[s][t] * e[s][c];
                e[t][c] = x;
            }
        }
        // state first (the next block waits for it), then this lane's outputs
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const float4 dd = DIAG ? load4(&bl.decay[4 * (rg + 8 * i)]) : make_float4(d0, d0, d0, d0);
            const float4 dl = DIAG ? load4(&bl.decay_lo[4 * (rg + 8 * i)]) : make_float4(d1, d1, d1, d1);
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                S[i][0][c] = fma2(f2(dd.x, dd.y), S[i][0][c], mul2(f2(dl.x, dl.y), S[i][0][c]));
                S[i][1][c] = fma2(f2(dd.z, dd.w), S[i][1][c], mul2(f2(dl.z, dl.w), S[i][1][c]));
            }
#pragma unroll
            for (int s = 0; s < BT; ++s) {
                const float4 bb = load4(&bl.b[s][4 * (rg + 8 * i)]);
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    S[i][0][c] = fma2(f2(bb.x, bb.y), f2(e[s][c]), S[i][0][c]);
                    S[i][1][c] = fma2(f2(bb.z, bb.w), f2(e[s][c]), S[i][1][c]);
                }
            }
        }
        const int t = rg >> 1;
        const float4 lq = load4(bl.tri[t]);
        float o[VL];
#pragma unroll
        for (int x = 0; x < VL; ++x) {
            auto mine = [&](int s) { return (rg & 1) ? e[s][VL + x] : e[s][x]; };
            o[x] = w[x] + lq.x * mine(0);
            o[x] += t >= 1 ? lq.y * mine(1) : 0.f;
            o[x] += t >= 2 ? lq.z * mine(2) : 0.f;
            o[x] += t >= 3 ? lq.w * mine(3) : 0.f;
        }
        if (t0 + t < len) {
            OUT *dst = op + (row0 + (size_t)(t0 + t) * stride) * D + c0 + (rg & 1) * VL;
            if constexpr (VL == 2) store2(dst, o[0], o[1]);
            else *dst = from_f32<OUT>(o[0]);
        }
    };

    __syncthreads();
    for (int st = 0; st < nst; ++st) {
#pragma unroll 1
        for (int m = 0; m < NW && (st * NW + m) * BT < len; ++m) process(stage[(st & 1) * NW + m], (st * NW + m) * BT);
        __syncthreads();   // one barrier per stage: the buffer written meanwhile is the one nobody reads
    }
    if (p.final_state) {
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < CPL; c += 2)
                    *reinterpret_cast<float2 *>(p.final_state + sbase + (size_t)(4 * (rg + 8 * i) + r) * D + c) =
                        (r & 1) ? make_float2(S[i][r >> 1][c].y, S[i][r >> 1][c + 1].y) : make_float2(S[i][r >> 1][c].x, S[i][r >> 1][c + 1].x);
    }
}

template <int D, int CPL, typename IO, typename OUT, bool DIAG>
cudaError_t launch_k(const TokenScanParams &p, cudaStream_t stream)
{
    auto kern = kla_token_scan_kernel<D, CPL, IO, OUT, DIAG>;
    constexpr int smem = 2 * NW * (int)sizeof(Block<D, CPL, DIAG>);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    kern<<<p.n_seq * p.H * (D / (NW * 4 * CPL)), 64 * NW, smem, stream>>>(p);
    count_launch(1);
    return cudaGetLastError();
}

template <int D, typename IO, typename OUT, bool DIAG>
cudaError_t launch_t(const TokenScanParams &p, cudaStream_t stream)
{
    if (p.n_seq * p.H == 0) return cudaSuccess;
    // 16 columns per warp as soon as that gives every SM more than two scanning warps (see the head of the file)
    if ((long long)p.n_seq * p.H * (D / 16) > 2LL * sm_count()) return launch_k<D, 4, IO, OUT, DIAG>(p, stream);
    return launch_k<D, 2, IO, OUT, DIAG>(p, stream);
}

template <int D, typename IO>
cudaError_t launch_io(const TokenScanParams &p, int out_dtype, cudaStream_t stream)
{
    if (out_dtype == KLA_BF16) return p.diag ? launch_t<D, IO, __nv_bfloat16, true>(p, stream) : launch_t<D, IO, __nv_bfloat16, false>(p, stream);
    return p.diag ? launch_t<D, IO, float, true>(p, stream) : launch_t<D, IO, float, false>(p, stream);
}

}  // namespace

cudaError_t launch_token_scan(const TokenScanParams &p, int d, int io_dtype, int out_dtype, cudaStream_t stream)
{
    if (d == 128) return io_dtype == KLA_BF16 ? launch_io<128, __nv_bfloat16>(p, out_dtype, stream) : launch_io<128, float>(p, out_dtype, stream);
    return io_dtype == KLA_BF16 ? launch_io<64, __nv_bfloat16>(p, out_dtype, stream) : launch_io<64, float>(p, out_dtype, stream);
}

}  // namespace kla
