// The product that the policy gradient's passes over node-state rows share: FP32 FMAs, one lane per output column,
// eight rows per warp.
#pragma once
#include "kernels.cuh"

namespace placeto {

constexpr int kRowWarps = 8, kRowThreads = 32 * kRowWarps;
constexpr int kRowsPerWarp = 8;

// acc[r][c] += in[r][0 .. K) . W[.][lane + 32 c], k ascending: W [K][D] and the rows in shared memory. K a multiple
// of 4 (zero padded). A weight load serves eight rows, a row's broadcast load four weights.
template <int D>
__device__ __forceinline__ void row_products(const float *W, const float *in, int stride, int K, int lane,
                                             float (&acc)[kRowsPerWarp][D / 32]) {
    constexpr int C = D / 32;
    for (int k = 0; k < K; k += 4) {
        float w[4][C];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < C; ++c) w[q][c] = W[(k + q) * D + lane + 32 * c];
#pragma unroll
        for (int r = 0; r < kRowsPerWarp; ++r) {
            const float4 x = *reinterpret_cast<const float4 *>(in + r * stride + k);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                acc[r][c] = fmaf(x.x, w[0][c], acc[r][c]);
                acc[r][c] = fmaf(x.y, w[1][c], acc[r][c]);
                acc[r][c] = fmaf(x.z, w[2][c], acc[r][c]);
                acc[r][c] = fmaf(x.w, w[3][c], acc[r][c]);
            }
        }
    }
}

}  // namespace placeto
