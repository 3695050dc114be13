// The blocked inverse of I + B X in shared memory, shared by the kernels that form it whole (chunk_wy.cu, bwd_chunk.cu).
#pragma once
#include "common.cuh"

namespace kla {

constexpr int LDT = 68;  // row stride (floats) of the fp32 solve matrix
constexpr int LDM = 40;  // row stride of a separate solve scratch

// One level of it (X strictly lower triangular, 64 x 64, in `tl`): for every pair of adjacent BS x BS diagonal blocks (T_00, T_11
// already inverted) the block below the diagonal becomes
//   T_10 = -T_11 (B_1 X_10 T_00).
// All pairs of the level are done at once by 256 threads, which `sync` joins: 32 result rows x BS columns, one 1 x 4 tile per
// thread; `mm` (row stride LDMM) holds the intermediate product.  T_11 is lower triangular: the columns k > r of its row r are
// skipped, by the thread or (UNIFORM) only where the whole warp can, so that trip counts are warp-uniform.
template <int BS, int LDMM, bool UNIFORM, typename Sync>
__device__ __forceinline__ void merge_level(float *tl, float *mm, const float *bet, int pt, Sync &&sync)
{
    constexpr int QPR = BS / 4;                 // column quads per row
    constexpr int RMASK = 128 / BS - 1;         // a warp covers 128 / BS consecutive rows
    const bool act = pt < 8 * BS;
    const int R = pt / QPR, c4 = (pt % QPR) * 4;
    const int pr = R / BS, r = R % BS;          // pair, row inside the block
    const int rb = (2 * pr + 1) * BS, cb = 2 * pr * BS;
    auto row_times = [](const float *a_row, const float *b, int ldb, int kend) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
        for (int k = 0; k < kend; k += 4) {
            const float4 a = load4(a_row + k);
            const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 x = load4(b + (k + u) * ldb);
                acc.x += av[u] * x.x; acc.y += av[u] * x.y; acc.z += av[u] * x.z; acc.w += av[u] * x.w;
            }
        }
        return acc;
    };
    if (act) {
        const float4 m = row_times(tl + (rb + r) * LDT + cb, tl + cb * LDT + cb + c4, LDT, BS);
        const float s = bet[rb + r];
        store4(&mm[R * LDMM + c4], make_float4(s * m.x, s * m.y, s * m.z, s * m.w));
    }
    sync();
    if (act) {
        const float4 t = row_times(tl + (rb + r) * LDT + rb, mm + (pr * BS) * LDMM + c4, LDMM, UNIFORM ? min(BS, (r | RMASK) + 1) : r + 1);
        store4(&tl[(rb + r) * LDT + cb + c4], make_float4(-t.x, -t.y, -t.z, -t.w));
    }
    sync();
}

}  // namespace kla
