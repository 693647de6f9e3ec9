// Interface between the sparse products (spmm.cu) and their tensor-core path
// (spmm_tc.cu), and the work of that path's first kernel: X is written out as
// three bf16 planes, and of W's rows is noted where each 64 columns begin.
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "split_bf16.cuh"

namespace csrt {

constexpr int kTcChunk = 64;        // columns of W (features) per step of the GEMM
constexpr int kTcGroup = 16;        // rows that a warp of the GEMM expands
constexpr int kTcMaxChunks = 256;   // (up to here the path was measured)
constexpr int32_t kTcNoColumn = 0x7fffffff;   // past the end of a row

// What the first kernel of an eligible product needs: if the matrix holds at
// least nnz_min entries it prepares both operands for the tensor-core kernel
// that follows, else it computes the product and that kernel leaves at once.
struct SpmmTcPrep {
    int64_t nnz_min;     // 0: no tensor-core kernel follows
    int32_t *start;      // [groups][chunks + 1][16] first entry of each row in each chunk
    __nv_bfloat16 *xp;   // [3][n][ld] the parts of X transposed
    int32_t k, ld, chunks;
    int32_t width;       // columns of X that a block of threads takes at a time
    int32_t vec;         // rows of X may be read as float4
    uint8_t *marks;      // [groups], then [chunks][ceil(n / width)] of X: 1: rows or values that the tensor cores can't take
    int32_t num_marks;
    uint32_t *cnt;       // [counters] of the tensor-core kernel's cut tiles, zeroed here: a kernel that gave up
    int32_t counters;    // waiting leaves nothing behind for the next call
};

struct SpmmTcPlan {
    SpmmTcPrep prep;
    CUtensorMap map_x;   // of prep.xp
    float *partial;
    int32_t n_tile, tiles_n, tiles, pairs;
    bool whole;   // no tile is shared by pairs
};

size_t spmm_tc_scratch_bytes(int32_t rows, int32_t cols, int32_t max_n);
// Fills the plan (prep.nnz_min > 0) if the product may run on the tensor cores.
// Everything that can fail is done here, before the product's first kernel is
// enqueued: a product that can't be planned runs on the sparse kernels alone.
// `units` and `t_entry` describe the sparse kernel: the work units its rows and
// entries are cut into, and its time per entry (microseconds).
void spmm_tc_plan(int32_t rows, int32_t k, int32_t n, int64_t capacity, const float *x, void *ws, size_t ws_bytes,
                  int32_t units, double t_entry, SpmmTcPlan *plan);
int spmm_tc_launch(const SpmmTcPlan &plan, const int32_t *row_ptr, const int32_t *col, const float *val, int32_t rows,
                   const float *x, int32_t n, float *y, const float *bias, int32_t relu, const float *mask, void *ws,
                   cudaStream_t s);

// X's planes of one chunk (64 features) and `width` columns (64 or 32) by a
// block of 256 threads: a lane holds the features 2 lane and 2 lane + 1 of its
// warp's eighth of the columns, read once. A value that can't be split marks
// the block (marks_w: the marks of W, before X's).
__device__ __forceinline__ void spmm_tc_prep_x(const SpmmTcPrep &a, const float *__restrict__ x, int32_t n, int chunk,
                                               int block, int marks_w) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = a.width / 8;
    const int c0 = block * a.width + warp * per;
    const int j0 = chunk * kTcChunk + lane * 2;
    float v[2][8];
    bool fits = true;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float *row = x + (int64_t)(j0 + h) * n;
#pragma unroll
        for (int e = 0; e < 8; e += 4) {
            const int c = c0 + e;
            if (j0 + h < a.k && a.vec && e < per && c < n) {   // (n is a multiple of 4 where rows may be read so)
                const float4 q = ldg_f4(row + c);
                v[h][e] = q.x; v[h][e + 1] = q.y; v[h][e + 2] = q.z; v[h][e + 3] = q.w;
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    v[h][e + i] = j0 + h < a.k && e < per && c + i < n ? __ldg(row + c + i) : 0.f;
            }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) fits &= split_fits(v[h][e]);
    }
    const int64_t plane = (int64_t)n * a.ld;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        if (e >= per || c0 + e >= n) break;
        __nv_bfloat162 p[3];
        split_bf16(make_float2(v[0][e], v[1][e]), p[0], p[1], p[2]);
        if (j0 < a.k) {   // (rows of the planes are multiples of 8 long: feature k may be written, as zero)
            __nv_bfloat162 *at = reinterpret_cast<__nv_bfloat162 *>(a.xp + (int64_t)(c0 + e) * a.ld + j0);
#pragma unroll
            for (int q = 0; q < 3; ++q) at[q * (plane / 2)] = p[q];
        }
    }
    const bool bad = __syncthreads_or(!fits);
    if (threadIdx.x == 0) a.marks[marks_w + chunk * ((n + a.width - 1) / a.width) + block] = bad;
}

// W's rows of one group of 16 by a block of 256 threads, two rows per warp.
// Columns ascend along a row, so its chunks are runs of entries, whose starts
// are stored (the entry whose predecessor lies in an earlier chunk). Rows whose
// columns don't ascend have no such runs, and of two entries of one column the
// operand could hold only one: their group is marked (the sparse kernels, which
// add up whatever a row stores, take any order). So is that of a value which
// can't be split.
__device__ __forceinline__ void spmm_tc_prep_w(const SpmmTcPrep &a, const int32_t *__restrict__ row_ptr,
                                               const int32_t *__restrict__ col, const float *__restrict__ val,
                                               int32_t rows, int32_t group) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the warp's two rows side by side, 128 entries of each per step, the next
    // step's on their way while this one's are worked on
    int32_t beg[2], end[2], len = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int32_t r = group * kTcGroup + warp * 2 + q;
        beg[q] = r < rows ? __ldg(row_ptr + r) : 0;
        end[q] = r < rows ? __ldg(row_ptr + r + 1) : 0;
        len = max(len, end[q] - beg[q]);
    }
    int32_t *start = a.start + (int64_t)group * (a.chunks + 1) * kTcGroup + warp * 2;
    int32_t c[2][4];
    float w[2][4];
    auto load = [&](int32_t i0) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int32_t i = beg[q] + i0 + h * 32 + lane;
                c[q][h] = i < end[q] ? __ldg(col + i) : kTcNoColumn;
                w[q][h] = i < end[q] ? __ldg(val + i) : 0.f;
            }
    };
    int before[2] = {-1, -1};   // column of the entry before this step's
    bool unfit = false;
    load(0);
    // (one step more than entries need ends every row: the chunks after its
    // last entry begin at its end)
    for (int32_t i0 = 0; i0 <= len; i0 += 128) {
        int32_t cc[2][4];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                cc[q][h] = c[q][h];
                unfit |= !split_fits(w[q][h]);
            }
        if (i0 + 128 <= len) load(i0 + 128);
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                int prev = __shfl_up_sync(0xffffffffu, cc[q][h], 1);
                if (lane == 0) prev = before[q];
                unfit |= cc[q][h] != kTcNoColumn && (cc[q][h] <= prev || cc[q][h] >= a.k);
                // mostly none or one (columns before `prev`: none)
                const int last = min(cc[q][h] >> 6, a.chunks);
                for (int ch = max(prev >> 6, -1) + 1; ch <= last; ++ch)
                    start[ch * kTcGroup + q] = min(beg[q] + i0 + h * 32 + lane, end[q]);
                before[q] = __shfl_sync(0xffffffffu, cc[q][h], 31);
            }
    }
    unfit = __syncthreads_or(unfit);
    if (threadIdx.x == 0) a.marks[group] = unfit;
}

// Both operands by a grid of 256-thread blocks: groups of W's rows (the longer
// pieces of work first), then X's blocks.
__device__ __forceinline__ void spmm_tc_prep(const SpmmTcPrep &a, const int32_t *__restrict__ row_ptr,
                                             const int32_t *__restrict__ col, const float *__restrict__ val,
                                             int32_t rows, const float *__restrict__ x, int32_t n) {
    const int nb = (n + a.width - 1) / a.width;
    const int ws = (rows + kTcGroup - 1) / kTcGroup, xs = a.chunks * nb;
    const int grid = (int)gridDim.x, b = (int)blockIdx.x;
    for (int i = b * blockDim.x + threadIdx.x; i < a.counters; i += grid * blockDim.x) a.cnt[i] = 0;
    for (int i = b; i < ws; i += grid) spmm_tc_prep_w(a, row_ptr, col, val, rows, i);
    // X by the blocks that had fewer groups to do
    const int busy = ws % grid, idle = grid - busy;
    if (busy && idle >= grid / 4) {
        if (b < busy) return;
        for (int i = b - busy; i < xs; i += idle) spmm_tc_prep_x(a, x, n, i / nb, i % nb, ws);
    } else {
        for (int i = b; i < xs; i += grid) spmm_tc_prep_x(a, x, n, i / nb, i % nb, ws);
    }
}

}  // namespace csrt
