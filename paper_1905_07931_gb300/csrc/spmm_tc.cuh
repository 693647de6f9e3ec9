// Interface between the sparse products (spmm.cu) and their tensor-core path
// (spmm_tc.cu), and the work of that path's first kernel: X is written out as
// two fp16 planes, W's entries are split likewise and sorted into the blocks
// in which the GEMM expands them.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>

#include "common.cuh"

namespace csrt {

constexpr int kTcChunk = 64;        // columns of W (features) per step of the GEMM
constexpr int kTcGroup = 16;        // rows whose entries of a chunk lie together
constexpr int kTcMaxChunks = 256;
constexpr int32_t kTcNoColumn = 0x7fffffff;   // past the end of a row

// What the first kernel of an eligible product needs: if the matrix holds at
// least nnz_min entries it prepares both operands for the tensor-core kernel
// that follows, else it computes the product and that kernel leaves at once.
struct SpmmTcPrep {
    int64_t nnz_min;     // 0: no tensor-core kernel follows
    uint32_t *parts;     // [capacity] high (bits 0-15) and low part of each entry, rows scaled by a power of two,
    uint16_t *place;     // and its byte offset in its group's 16 x 128 byte block of the GEMM's operand
    int32_t *start;      // [groups][chunks + 1] first entry of each group's chunk
    float *wscale;       // [rows] undoes the rows' scale
    __half *xp;          // [2][n][ld] high and low parts of X transposed, scaled per chunk and `width` columns
    float *xscale;       // [chunks][ceil(n / width)] undoes that
    int32_t k, ld, chunks, width;
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

// Values a factor may take on the tensor-core path (products and sums of
// these stay far inside float32's range). With larger ones, infinities or NaN
// the whole product is gathered instead: it then costs about what the sparse
// kernel would.
constexpr uint32_t kTcLimitBits = (127u + 50u) << 23;   // 2^50

// The power of two that brings a value of magnitude bits `mx` into [2^14,
// 2^15) (the top of fp16's range) and the one that undoes it. Magnitudes
// below 2^-100 are scaled as 2^-100.
__device__ __forceinline__ void fp16_scales(uint32_t mx, float &down, float &up) {
    const uint32_t ex = max(mx >> 23, 27u);
    down = __uint_as_float((268u - ex) << 23);   // 2^(14 - (ex - 127))
    up = __uint_as_float((ex - 14u) << 23);      // 2^((ex - 127) - 14)
}
// High and low part of a scaled value: v = hi + lo * 2^-11, 22 to 23 bits.
__device__ __forceinline__ void fp16_split(float v, __half &hi, __half &lo) {
    hi = __float2half_rn(v);
    lo = __float2half_rn((v - __half2float(hi)) * 2048.f);
}

// Byte offset of column j of row r in a block of 16 rows of 128 bytes with
// the 128-byte swizzle.
__device__ __forceinline__ uint32_t tc_place(int r, int j) {
    return (uint32_t)(r * 128 + (((j >> 3) ^ (r & 7)) << 4) + (j & 7) * 2);
}

// X's planes of one chunk (64 features) and `width` columns (64 or 32), which
// share a scale (marks_w: the marks of W before X's): a block of 256 threads, a lane holds the features j and j +
// 32 of its warp's eighth of the columns, read once. s_max: 8 words.
__device__ __forceinline__ void spmm_tc_prep_x(const SpmmTcPrep &a, const float *__restrict__ x, int32_t n, int chunk,
                                               int block, int marks_w, uint32_t *s_max) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = a.width / 8;
    const int c0 = block * a.width + warp * per;
    float v[2][8];
    uint32_t mx = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t j = (int64_t)chunk * kTcChunk + h * 32 + lane;
        const float *row = x + j * n;
#pragma unroll
        for (int e = 0; e < 8; e += 4) {
            const int c = c0 + e;
            if (j < a.k && a.vec && e < per && c < n) {   // (n is a multiple of 4 where rows may be read so)
                const float4 q = ldg_f4(row + c);
                v[h][e] = q.x; v[h][e + 1] = q.y; v[h][e + 2] = q.z; v[h][e + 3] = q.w;
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) v[h][e + i] = j < a.k && e < per && c + i < n ? __ldg(row + c + i) : 0.f;
            }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) mx = max(mx, __float_as_uint(v[h][e]) & 0x7fffffffu);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) s_max[warp] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) mx = max(mx, s_max[w]);
    __syncthreads();   // s_max is free again
    const bool bad = mx >= kTcLimitBits;   // infinities and NaN too
    float down, up;
    fp16_scales(mx, down, up);
    if (threadIdx.x == 0) {
        const int at = chunk * ((n + a.width - 1) / a.width) + block;
        a.marks[marks_w + at] = bad;
        a.xscale[at] = up;
    }
    if (bad) return;
    const int64_t plane = (int64_t)n * a.ld;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        if (e >= per || c0 + e >= n) break;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = chunk * kTcChunk + h * 32 + lane;
            if (j >= a.k) continue;
            __half hi, lo;
            fp16_split(v[h][e] * down, hi, lo);
            __half *p = a.xp + (int64_t)(c0 + e) * a.ld + j;
            p[0] = hi;
            p[plane] = lo;
        }
    }
}

// W's entries of one group of 16 rows by a block of 256 threads, two rows per
// warp. The group's entries keep their range of the CSR arrays, sorted by
// chunk and then by row. Columns ascend along a row, so its chunks are runs:
// a first pass notes where each begins (the entry whose predecessor lies in
// an earlier chunk) and each row's largest magnitude; the rows' counts of
// each chunk, added up, give every run its place, kept as the difference
// from its place in the CSR; the second pass splits the entries and stores
// them. tab: [chunks + 1][17] words (17: rows of one chunk in different banks).
// Rows whose columns don't ascend have no such runs, and of two entries of one
// column the operand could hold only one: their group is marked and left (the
// sparse kernels, which add up whatever a row stores, take any order).
__device__ __forceinline__ void spmm_tc_prep_w(const SpmmTcPrep &a, const int32_t *__restrict__ row_ptr,
                                               const int32_t *__restrict__ col, const float *__restrict__ val,
                                               int32_t rows, int32_t group, int32_t (*tab)[17]) {
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
    uint32_t mx[2] = {0, 0};
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
                mx[q] = max(mx[q], __float_as_uint(w[q][h]) & 0x7fffffffu);
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
                    tab[ch][warp * 2 + q] = min(i0 + h * 32 + lane, end[q] - beg[q]);
                before[q] = __shfl_sync(0xffffffffu, cc[q][h], 31);
            }
    }
    load(0);
    float down[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int32_t r = group * kTcGroup + warp * 2 + q;
        const uint32_t m = __reduce_max_sync(0xffffffffu, mx[q]);
        unfit |= m >= kTcLimitBits;   // (infinities and NaN too)
        float up;
        fp16_scales(m, down[q], up);
        if (lane == 0 && r < rows) a.wscale[r] = up;
    }
    __shared__ int32_t s_sum[9];
    const int32_t base = __ldg(row_ptr + group * kTcGroup);
    unfit = __syncthreads_or(unfit);
    if (threadIdx.x == 0) a.marks[group] = unfit;
    if (unfit) return;
    // thread = chunk: its rows' counts, the chunks' first entries by a block scan
    {
        const int ch = threadIdx.x;
        int32_t n = 0;
        if (ch < a.chunks) {
#pragma unroll
            for (int r = 0; r < kTcGroup; ++r) n += tab[ch + 1][r] - tab[ch][r];
        }
        int32_t incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_sum[warp] = incl;
        // (each thread reads its successor's row of tab: all before any writes)
        int32_t cnt[kTcGroup];
#pragma unroll
        for (int r = 0; r < kTcGroup; ++r) cnt[r] = ch < a.chunks ? tab[ch + 1][r] - tab[ch][r] : 0;
        __syncthreads();
        int32_t at = base + incl - n;
#pragma unroll
        for (int o = 0; o < 8; ++o)
            if (o < warp) at += s_sum[o];
        int32_t *out = a.start + (int64_t)group * (a.chunks + 1);
        if (ch < a.chunks) {
            out[ch] = at;
#pragma unroll
            for (int r = 0; r < kTcGroup; ++r) {
                tab[ch][r] = at - tab[ch][r];   // place of the row's entry i: tab + i
                at += cnt[r];
            }
            if (ch == a.chunks - 1) out[a.chunks] = at;
        }
    }
    __syncthreads();
    for (int32_t i0 = 0; i0 < len; i0 += 128) {
        int32_t cc[2][4];
        float ww[2][4];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                cc[q][h] = c[q][h];
                ww[q][h] = w[q][h];
            }
        if (i0 + 128 < len) load(i0 + 128);
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                if (cc[q][h] == kTcNoColumn) continue;
                __half hi, lo;
                fp16_split(ww[q][h] * down[q], hi, lo);
                const int32_t p = tab[cc[q][h] >> 6][warp * 2 + q] + i0 + h * 32 + lane;
                a.parts[p] = (uint32_t)__half_as_ushort(hi) | (uint32_t)__half_as_ushort(lo) << 16;
                a.place[p] = (uint16_t)tc_place(warp * 2 + q, cc[q][h] & 63);
            }
    }
    __syncthreads();   // tab is free again
}

// Both operands by a grid of 256-thread blocks: groups of W's rows (the longer
// pieces of work first), then X's blocks.
__device__ __forceinline__ void spmm_tc_prep(const SpmmTcPrep &a, const int32_t *__restrict__ row_ptr,
                                             const int32_t *__restrict__ col, const float *__restrict__ val,
                                             int32_t rows, const float *__restrict__ x, int32_t n) {
    __shared__ uint32_t s_max[8];
    extern __shared__ int32_t s_tab[][17];   // [chunks + 1], allocated only where this path may run
    const int nb = (n + a.width - 1) / a.width;
    const int ws = (rows + kTcGroup - 1) / kTcGroup, xs = a.chunks * nb;
    const int grid = (int)gridDim.x, b = (int)blockIdx.x;
    for (int i = b * blockDim.x + threadIdx.x; i < a.counters; i += grid * blockDim.x) a.cnt[i] = 0;
    for (int i = b; i < ws; i += grid) spmm_tc_prep_w(a, row_ptr, col, val, rows, i, s_tab);
    // X by the blocks that had fewer groups to do
    const int busy = ws % grid, idle = grid - busy;
    if (busy && idle >= grid / 4) {
        if (b < busy) return;
        for (int i = b - busy; i < xs; i += idle) spmm_tc_prep_x(a, x, n, i / nb, i % nb, ws, s_max);
    } else {
        for (int i = b; i < xs; i += grid) spmm_tc_prep_x(a, x, n, i / nb, i % nb, ws, s_max);
    }
}

}  // namespace csrt
