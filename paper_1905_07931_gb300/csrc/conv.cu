// Convolution with a compressed (CSR) filter bank, without the unfolded input.
//
// Section 3.2 lowers a convolution to the product of the filter matrix W
// (C_out x C_in*k*k, here in CSR) with the unfolded input (the Caffe
// im2col matrix, C_in*k*k x B*Ho*Wo). The forward pass only needs, for each
// output pixel, the stored filter taps of its channel applied to the input
// window, so this kernel reads the input in place: the unfolded matrix, which
// is k*k times larger than the input, is never written or read.
//
// One block per (tile of output pixels, group of output channels). A block
// stages the taps of its channels in shared memory as (input offset, weight)
// pairs: tap t = (c*k + ky)*k + kx of a CSR row reads input pixel
// x[c][b][oy+ky][ox+kx], c*B*H*W + ky*W + kx elements from the window's
// corner x[0][b][oy][ox]. Each thread accumulates its output pixels over the
// taps of one channel after the other in CSR order, with one fused
// multiply-add per tap, then applies the bias and ReLU. A window is reused by
// all taps of all channels of the block from L1.
//
// What bounds it: instruction issue (75% to 86% of its slots) and the L1 reads
// (78% to 82%), one add, one load and one multiply-add per tap and pixel. Dividing a pixel number into sample, row and column in 64
// bits for every channel took more time than the taps of a layer with few of
// them, so the channels of a group share the corners, and inputs under 4 GiB
// (every one of practical size) use 32-bit offsets. LeNet-5 at 1000 images:
// conv1 (20 channels, 7.9 taps each) 61.1 -> 29.4 us; conv2 (50 channels, 42
// taps) 51.5 -> 41.3 us, and 36.2 us with the lane order below; with one output
// pointer per thread that moves on by a channel, and the pixels of a whole
// tile unchecked, 27.0 and 35.8 us. Taps unrolled by 1, 2, 4, 8: conv1 27.6,
// 27.6, 27.0, 27.7 us, conv2 40.7, 36.4, 35.8, 36.4 us.
//
// Lane order: a warp that reads 32 / Wo consecutive output rows for one tap
// touches rows W words apart, which share banks unless W is a multiple of Wo.
// Where Wo divides 32, the warp takes rows 2^e apart instead, with the
// smallest e <= 3 that makes (W << e) an odd multiple of Wo modulo 32: its
// reads then fall into 32 different banks (W = 12, Wo = 8, rows 0 2 4 6: conv2
// 41.3 -> 36.1 us; 32 x 32 channels of 20 x 20, Wo = 16: 86.7 -> 69.9 us). The
// warps of a block take the rows between, so the pixels of a block and the sum
// of each pixel are the same as without.
#include "common.cuh"

namespace csrt {

constexpr int kConvThreads = 256;
constexpr int kConvPer = 4;          // output pixels per thread, large outputs
constexpr int kConvTaps = 1024;      // taps staged per round
constexpr int kConvGroup = 32;       // most output channels per block
constexpr int kConvBlocksPerSM = 16;  // blocks per SM to keep when channels share a block

template <typename I>
struct ConvTap {
    I off;     // bytes from a window's corner to the tap's input
    float w;
};

// I: uint32_t when the input's bytes and the pixel count fit, else uint64_t.
template <typename I, int kPer>
__global__ void __launch_bounds__(kConvThreads) conv_sparse_fwd_kernel(
    const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col, const float *__restrict__ val, int32_t rows,
    int32_t group, int32_t ox_bits, int32_t step_bits, const float *__restrict__ x, int32_t b, int32_t h, int32_t w, int32_t k,
    const float *__restrict__ bias, int32_t relu, float *__restrict__ y) {
    pdl_enter();
    __shared__ ConvTap<I> s_tap[kConvTaps];
    __shared__ int32_t s_end[kConvGroup];
    const I ho = h - k + 1, wo = w - k + 1;
    const I plane = (I)b * h * w;              // one input channel
    const I npix = (I)b * ho * wo;             // output pixels per channel
    const int m0 = blockIdx.y * group, m1 = imin(m0 + group, rows);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int step_mask = (1 << step_bits) - 1, ox_mask = (1 << ox_bits) - 1;
    // the thread's place in its block's pixels: the lane order described above
    const int t = (lane & ox_mask) | (warp & step_mask) << ox_bits | (lane >> ox_bits) << (ox_bits + step_bits) |
                  (warp >> step_bits) << (5 + step_bits);
    const I p0 = (I)blockIdx.x * (kConvThreads * kPer) + t;
    I corner[kPer];   // bytes to the window corner of each pixel; past the last pixel, of pixel 0
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const I p = p0 + q * kConvThreads;
        const I pp = p < npix ? p : 0;
        const I s = pp / (ho * wo);
        const I rem = pp - s * (ho * wo);
        const I oy = rem / wo, ox = rem - oy * wo;
        corner[q] = ((s * h + oy) * w + ox) * 4;
    }
    // one pointer for all channels: a whole tile's stores need no address or check
    float *yp = y + ((int64_t)m0 * (int64_t)npix + (int64_t)p0);
    const bool full = p0 + (kPer - 1) * kConvThreads < npix;
    const int32_t t0 = __ldg(row_ptr + m0), t1 = __ldg(row_ptr + m1);
    if ((int)threadIdx.x < m1 - m0) s_end[threadIdx.x] = __ldg(row_ptr + m0 + threadIdx.x + 1);
    float acc[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) acc[q] = 0.f;
    int m = m0;
    for (int32_t tb = t0;; tb += kConvTaps) {
        const int nt = imin(kConvTaps, t1 - tb);
        const bool last = t1 - tb <= kConvTaps;
        __syncthreads();   // the previous round's taps are consumed
        for (int i = threadIdx.x; i < nt; i += kConvThreads) {
            const int tap = __ldg(col + tb + i);
            const int c = tap / (k * k), kk = tap - c * k * k;
            const int ky = kk / k, kx = kk - ky * k;
            s_tap[i] = {((I)c * plane + (I)ky * w + kx) * 4, __ldg(val + tb + i)};
        }
        __syncthreads();
        for (int i = 0; m < m1; ++m) {
            const int end = s_end[m - m0] - tb;
            const int stop = imin(end, nt);
#pragma unroll 4
            for (; i < stop; ++i) {
                const ConvTap<I> tap = s_tap[i];
#pragma unroll
                for (int q = 0; q < kPer; ++q)
                    acc[q] = fmaf(tap.w, __ldg((const float *)((const char *)x + (I)(corner[q] + tap.off))), acc[q]);
            }
            if (end > nt && !last) break;   // the channel's taps go on in the next round
            const float bm = bias ? __ldg(bias + m) : 0.f;
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                float v = acc[q];
                acc[q] = 0.f;
                if (bias) v = __fadd_rn(v, bm);
                if (relu) v = fmaxf(v, 0.f);
                if (full || p0 + q * kConvThreads < npix) yp[q * kConvThreads] = v;
            }
            yp += npix;
        }
        if (last) break;
    }
}

}  // namespace csrt

using namespace csrt;

extern "C" int csrt_conv2d_sparse_fwd(const csrt_csr *w, const float *x, int32_t c, int32_t b, int32_t h,
                                      int32_t wd, int32_t k, const float *bias, int32_t relu, float *y,
                                      void *stream) {
    CSRT_ARG(w != nullptr && w->row_ptr != nullptr, "csr is NULL");
    CSRT_ARG(c > 0 && b >= 0 && k > 0 && h >= k && wd >= k, "bad convolution shape");
    CSRT_ARG(w->cols == c * k * k, "filter matrix has %d columns, expected C*k*k = %d", w->cols, c * k * k);
    CSRT_ARG(w->rows > 0 && w->rows <= 65535, "output channels must be in 1..65535");
    const int64_t npix = (int64_t)b * (h - k + 1) * (wd - k + 1);
    if (npix == 0) return CSRT_OK;
    CSRT_ARG(x != nullptr && y != nullptr, "x or y is NULL");
    CSRT_ARG(w->capacity == 0 || (w->col_idx && w->val), "col_idx/val NULL");
    const int64_t tiles4 = ceil_div<int64_t>(npix, (int64_t)kConvThreads * kConvPer);
    CSRT_ARG(tiles4 < ((int64_t)1 << 31), "too many output pixels");
    // byte offsets in 32 bits; the pixel numbers of the last tile run past npix by less than a tile
    const bool narrow = (int64_t)c * b * h * wd < ((int64_t)1 << 30) && npix < ((int64_t)1 << 31);
    // Four pixels per thread share the staged taps and keep four loads in
    // flight; with fewer than two blocks per SM, one pixel per thread spreads
    // the work over more threads instead (conv2 of LeNet-5 at 64 images, 200
    // blocks: 7.8 us with four, 6.2 us with one; conv1 at 64, 720 blocks: 4.9 us
    // with four, 7.3 us with one).
    const bool small = narrow && tiles4 * w->rows < (int64_t)num_sms() * 2;
    const int64_t tiles = small ? ceil_div<int64_t>(npix, kConvThreads) : tiles4;
    // As many channels per block as leave kConvBlocksPerSM blocks per SM
    // (conv1 / conv2 of LeNet-5 at 1000 images with 8, 16 and 32 per SM: 26.9 /
    // 46.6, 27.5 / 40.8, 30.6 / 40.7 us).
    const int group = (int)imax<int64_t>(
        1, imin<int64_t>(kConvGroup, tiles * w->rows / ((int64_t)num_sms() * kConvBlocksPerSM)));
    int ox_bits = 5, step_bits = 0;   // consecutive pixels in consecutive lanes
    const int wo = wd - k + 1;
    if (wo < 32 && 32 % wo == 0)
        for (int e = 0; e <= 3; ++e)
            if (((int64_t)wd << e) % (2 * wo) == wo) {
                while ((1 << ox_bits) > wo) --ox_bits;
                step_bits = e;
                break;
            }
    const auto kern = small ? conv_sparse_fwd_kernel<uint32_t, 1>
                      : narrow ? conv_sparse_fwd_kernel<uint32_t, kConvPer> : conv_sparse_fwd_kernel<uint64_t, kConvPer>;
    launch_pdl(kern, dim3((unsigned)tiles, (unsigned)ceil_div(w->rows, group)), dim3(kConvThreads), 0,
               as_stream(stream), w->row_ptr, w->col_idx, w->val, w->rows, group, ox_bits, step_bits, x, b, h, wd, k,
               bias, relu, y);
    count_launch();
    return check_launch("conv_sparse_fwd_kernel");
}
