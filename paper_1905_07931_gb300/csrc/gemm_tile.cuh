// One 64 x 64 tile of G = dY X^T by 256 threads with float32 multiply-adds: the
// body of the CUDA-core gradient kernel (gemm.cu), which the tensor-core one
// (gemm_split.cu) also runs for operands that it can't split.
#pragma once

#include "common.cuh"

namespace csrt {

constexpr int kGBM = 64, kGBN = 64, kGBK = 16;
struct GemmTileSmem {
    float as[kGBK][kGBM + 4];
    float bs[kGBK][kGBN + 4];
};

// Rows i0.. and columns j0.. of the sum over columns nb <= c < ne, one chain
// per element in the order of c, to slice `slice` of out ([.][m][k]). tid:
// 0..255; sync(): a barrier of the 256.
template <typename Sync>
__device__ __forceinline__ void gemm_nt_tile(const float *__restrict__ dy, const float *__restrict__ x, int32_t m,
                                             int32_t k, int32_t n, int nb, int ne, int64_t i0, int64_t j0, int tid,
                                             GemmTileSmem &s, float *__restrict__ out, int slice, Sync sync) {
    const int ty = tid / 16, tx = tid % 16;
    float acc[4][4] = {};
    for (int c0 = nb; c0 < ne; c0 += kGBK) {
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const int idx = tid + l * 256;
            const int r = idx / kGBK, kk = idx % kGBK;
            const int c = c0 + kk;
            s.as[kk][r] = (i0 + r < m && c < ne) ? __ldg(dy + (i0 + r) * n + c) : 0.f;
            s.bs[kk][r] = (j0 + r < k && c < ne) ? __ldg(x + (j0 + r) * n + c) : 0.f;
        }
        sync();
#pragma unroll
        for (int kk = 0; kk < kGBK; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                a[t] = s.as[kk][ty * 4 + t];
                b[t] = s.bs[kk][tx * 4 + t];
            }
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(a[p], b[q], acc[p][q]);
        }
        sync();
    }
    float *o = out + (int64_t)slice * m * k;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const int64_t i = i0 + ty * 4 + p;
        if (i >= m) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t j = j0 + tx * 4 + q;
            if (j < k) o[i * k + j] = acc[p][q];
        }
    }
}

}  // namespace csrt
