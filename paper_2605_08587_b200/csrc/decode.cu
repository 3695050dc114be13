// Recurrent decode step (Algorithm 1, left panel; Eq. 3) -- memory-bound kernel.
//
// One warp owns 16 consecutive d_v columns of one head's d_k x d_v fp32 state: a lane 4 of them over d_k / 8 rows.  Columns evolve
// independently (the rank-one write is k e^T), so no warp talks to another and nothing waits at a barrier.  The slice is read
// from HBM exactly once (whole 32-byte sectors), kept in registers, and written back once:
//
//   a = S^T k, c = S^T q                       (one sweep over the registers)
//   e = v - alpha a,  beta = eta / (||k||^2 + eps)
//   S <- alpha S + beta k e^T                  (written back)
//   o = S_new^T q = alpha c + beta (k.q) e     (no second sweep over the state)
//
// Several steps in one call keep the slice in registers from the first to the last: one launch per step read and wrote the
// state every time (four steps at B = 512, H = 8, d = 128: 337 us for 4 x 554 MB).  What bounds several steps is the latency of a
// step times the steps: with 32 columns to a block of four warps, whose sums crossed the warps in shared memory behind two
// barriers, those four steps took 163 us (83 us of it the memory traffic), now 125; with 8 columns (half a 64-byte segment of a row per
// request) 138, and a single step on 64 sequences 13.0 instead of 11.6 us.
//
// Diagonal gates (one decay per row of the state, DIAG): the decayed vectors alpha o k and alpha o q stand in the sweep, so
// a = S^T (alpha o k) and c = S^T (alpha o q) come out decayed already; everything else is the same.  (The whole-sequence
// scan with one token took 24.8 us at B = 64, H = 8, d = 128: eight-column warps, operands requested three tokens ahead of a
// loop of one; now 11.9 us.)
#include "common.cuh"
#include "scan_pieces.cuh"

namespace kla {

// N consecutive elements as loaded (16-byte pieces), converted on use.
template <typename IO, int N>
struct Row {
    float4 r[N / 4];
    __device__ __forceinline__ void load(const float *p)
    {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) r[i] = load4(p + 4 * i);
    }
    __device__ __forceinline__ void get(float (&x)[N]) const
    {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) { x[4 * i] = r[i].x; x[4 * i + 1] = r[i].y; x[4 * i + 2] = r[i].z; x[4 * i + 3] = r[i].w; }
    }
};
template <int N>
struct Row<__nv_bfloat16, N> {
    uint2 r[N / 4];
    __device__ __forceinline__ void load(const __nv_bfloat16 *p)
    {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) r[i] = *reinterpret_cast<const uint2 *>(p + 4 * i);
    }
    __device__ __forceinline__ void get(float (&x)[N]) const
    {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            x[4 * i] = __uint_as_float(r[i].x << 16); x[4 * i + 1] = __uint_as_float(r[i].x & 0xffff0000u);
            x[4 * i + 2] = __uint_as_float(r[i].y << 16); x[4 * i + 3] = __uint_as_float(r[i].y & 0xffff0000u);
        }
    }
};

template <int D, typename IO, typename OUT, bool DIAG>
__global__ void __launch_bounds__(128, 4) kla_decode_kernel(DecodeParams p)
{
    constexpr int NP = D / 8;   // rows of a lane
    const int unit = blockIdx.x * 4 + (threadIdx.x >> 5);   // (sequence and head, 16 columns)
    const int bh = unit / (D / 16), lane = threadIdx.x & 31;
    const int col = (unit % (D / 16)) * 16 + (lane & 3) * 4, row0 = (lane >> 2) * NP;

    // The kernel is launched with programmatic stream serialisation, so it may start while the previous kernel on the stream
    // drains; everything it reads may be that kernel's output.
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // 1. the vectors of one token: requested a step ahead (a use, even a conversion, would wait for them)
    const IO *qp = reinterpret_cast<const IO *>(p.q) + (size_t)bh * D + row0;
    const IO *kp = reinterpret_cast<const IO *>(p.k) + (size_t)bh * D + row0;
    const IO *vp = reinterpret_cast<const IO *>(p.v) + (size_t)bh * D + col;
    OUT *op = reinterpret_cast<OUT *>(p.out) + (size_t)bh * D + col;
    Row<IO, NP> k_raw, q_raw;
    Row<float, DIAG ? NP : 4> la_row;
    Vec4<IO> v_raw;
    float la_raw = 0.f, eta = 0.f;
    auto request = [&](size_t step) {
        const size_t row = step * (size_t)p.BH;
        k_raw.load(kp + row * D);
        q_raw.load(qp + row * D);
        if constexpr (DIAG) la_row.load(p.log_alpha + (row + bh) * D + row0);
        else la_raw = p.log_alpha[row + bh];
        eta = p.eta[row + bh];
        v_raw.load(vp + row * D);
    };
    request(0);

    // 2. the state; then let the next kernel on the stream start (it waits before it reads)
    float *Sp = p.state + (size_t)bh * D * D + (size_t)row0 * D + col;
    float2 s[NP][2];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const float4 x = load4(Sp + (size_t)i * D);
        s[i][0] = f2(x.x, x.y);
        s[i][1] = f2(x.z, x.w);
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

#pragma unroll 1
    for (int step = 0; step < (DIAG ? 1 : p.n_steps); ++step) {
        float kr[NP], ar[NP];
        float kk = 0.f, kq = 0.f, qq = 0.f, alpha = 1.f;
        float2 a2[2] = {f2(0.f), f2(0.f)}, c2[2] = {f2(0.f), f2(0.f)};
        {
            float qr[NP];
            k_raw.get(kr);
            q_raw.get(qr);
            if constexpr (DIAG) {
                la_row.get(ar);
#pragma unroll
                for (int i = 0; i < NP; ++i) ar[i] = expf(ar[i]);
            } else {
                alpha = expf(la_raw);
            }
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                kk += kr[i] * kr[i];
                kq += kr[i] * qr[i];
                if (p.qnorm) qq += qr[i] * qr[i];
                // 3. a = S^T k and c = S^T q over this lane's rows, two columns to an instruction
                const float2 kd = f2(DIAG ? ar[i] * kr[i] : kr[i]), qd = f2(DIAG ? ar[i] * qr[i] : qr[i]);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    a2[e] = fma2(s[i][e], kd, a2[e]);
                    c2[e] = fma2(s[i][e], qd, c2[e]);
                }
            }
        }
        const float eta_now = eta;
        const float4 vv = v_raw.get();
        if (!DIAG && step + 1 < p.n_steps) request((size_t)step + 1);
        // Sums over the 8 row groups (lanes equal modulo 4), by halving: lane bits 4, 3, 2 choose between a and c and the column
        const bool b16 = lane & 16, b8 = lane & 8, b4 = lane & 4;
        float x[4] = {b16 ? c2[0].x : a2[0].x, b16 ? c2[0].y : a2[0].y, b16 ? c2[1].x : a2[1].x, b16 ? c2[1].y : a2[1].y};
        {
            const float y[4] = {b16 ? a2[0].x : c2[0].x, b16 ? a2[0].y : c2[0].y, b16 ? a2[1].x : c2[1].x, b16 ? a2[1].y : c2[1].y};
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] += __shfl_xor_sync(0xffffffffu, y[i], 16);
        }
        float z[2] = {b8 ? x[2] : x[0], b8 ? x[3] : x[1]};
        z[0] += __shfl_xor_sync(0xffffffffu, b8 ? x[0] : x[2], 8);
        z[1] += __shfl_xor_sync(0xffffffffu, b8 ? x[1] : x[3], 8);
        float ac = b4 ? z[1] : z[0];
        ac += __shfl_xor_sync(0xffffffffu, b4 ? z[0] : z[1], 4);   // a or c of column (b8, b4)
#pragma unroll
        for (int o = 16; o > 2; o >>= 1) {
            kk += __shfl_xor_sync(0xffffffffu, kk, o);
            kq += __shfl_xor_sync(0xffffffffu, kq, o);
            if (p.qnorm) qq += __shfl_xor_sync(0xffffffffu, qq, o);
        }

        // 4. residual, coefficient, update, read-out
        const float beta = p.coeff_eta ? eta_now : eta_now / (kk + p.eps);   // Eq. 3, or the gated-delta-rule coefficient
        const int src = lane & 3;
        const float e[4] = {vv.x - alpha * __shfl_sync(0xffffffffu, ac, src), vv.y - alpha * __shfl_sync(0xffffffffu, ac, src | 4),
                            vv.z - alpha * __shfl_sync(0xffffffffu, ac, src | 8), vv.w - alpha * __shfl_sync(0xffffffffu, ac, src | 12)};
        const float2 e2[2] = {f2(e[0], e[1]), f2(e[2], e[3])};
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const float2 bk = f2(beta * kr[i]), al = f2(DIAG ? ar[i] : alpha);
#pragma unroll
            for (int h = 0; h < 2; ++h) s[i][h] = fma2(bk, e2[h], mul2(al, s[i][h]));
        }
        if (b16) {   // the lanes that hold c
            const float rn = p.qnorm ? 1.f / sqrtf(qq) : 1.f;   // read-out over ||q|| (Algorithm 1 left) when asked for
            const float ej = b8 ? (b4 ? e[3] : e[2]) : (b4 ? e[1] : e[0]);
            op[(size_t)step * p.BH * D + (b8 ? 2 : 0) + (b4 ? 1 : 0)] = from_f32<OUT>(rn * (alpha * ac + beta * kq * ej));
        }
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) store4(Sp + (size_t)i * D, make_float4(s[i][0].x, s[i][0].y, s[i][1].x, s[i][1].y));
}

template <int D, typename IO, typename OUT, bool DIAG>
static cudaError_t launch_decode_k(const DecodeParams &p, cudaStream_t stream)
{
    // programmatic dependent launch: the kernel's prologue may start while the previous kernel on the stream
    // drains; its state accesses come after griddepcontrol.wait
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.BH * (D / 64)));
    cfg.blockDim = dim3(128);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kla_decode_kernel<D, IO, OUT, DIAG>, p);
    count_launch(1);
    return err != cudaSuccess ? err : cudaGetLastError();
}

template <int D, typename IO, typename OUT>
static cudaError_t launch_decode_t(const DecodeParams &p, cudaStream_t stream)
{
    return p.diag ? launch_decode_k<D, IO, OUT, true>(p, stream) : launch_decode_k<D, IO, OUT, false>(p, stream);
}

cudaError_t launch_decode(const DecodeParams &p, int d, int io_dtype, int out_dtype, cudaStream_t stream)
{
    const int key = (d == 128 ? 4 : 0) | (io_dtype == KLA_BF16 ? 2 : 0) | (out_dtype == KLA_BF16 ? 1 : 0);
    switch (key) {
        case 0: return launch_decode_t<64, float, float>(p, stream);
        case 1: return launch_decode_t<64, float, __nv_bfloat16>(p, stream);
        case 2: return launch_decode_t<64, __nv_bfloat16, float>(p, stream);
        case 3: return launch_decode_t<64, __nv_bfloat16, __nv_bfloat16>(p, stream);
        case 4: return launch_decode_t<128, float, float>(p, stream);
        case 5: return launch_decode_t<128, float, __nv_bfloat16>(p, stream);
        case 6: return launch_decode_t<128, __nv_bfloat16, float>(p, stream);
        default: return launch_decode_t<128, __nv_bfloat16, __nv_bfloat16>(p, stream);
    }
}

}  // namespace kla
