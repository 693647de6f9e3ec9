// Dense weight gradient G = dY X^T in float32 accuracy on the tensor cores.
//
// Every float32 factor is the sum of three bf16 parts, all of its 24 bits at
// every exponent below 2^28; six of the nine products of parts are taken, the
// large one in sums of 64 columns that are added up with round to nearest
// (split_bf16.cuh). The error against 64 bits is below that of a chain of fused
// multiply-adds over the same columns (N(0, 1) over 256 columns 0.8e-7 against
// 2.9e-7, positive factors 0.9e-7 against 2.5e-7, ReLU features and errors that
// came through a ReLU 0.5e-7 against 1.4e-7), and where a single sample makes
// up a sum, one rounding and the parts left out, 1.1e-7 at most against 6.0e-8.
// (With one accumulator for all six products that was 1.6e-7, and parts that
// are not scaled lost bits of values under 2^-110.)
//
//  split_rows_kernel       dY and X to their planes (bf16, [3][rows][ld]) in the
//                          workspace, a warp per row; blocks of eight rows that hold
//                          a value of 2^28 or more, an infinity or a NaN are marked.
//  gemm_split_kernel       CTA pairs (cta_group::2) walk 256 x 256 tiles of G:
//                          per 64 columns six 16 KB slices per CTA (three planes
//                          of its 128 rows of dY and 128 rows of X) by TMA, 20
//                          MMAs of M = 256, N = 256, K = 16 for the small products
//                          and 4 for x1 y1, each kind with an accumulator of its
//                          own in tensor memory; while the next columns' 20 run,
//                          sixteen warps per CTA read x1 y1 back and add it to the
//                          sums of their 32 rows x 64 columns in registers.
// With any block marked the second kernel computes all of G in tiles of float32
// multiply-adds instead (gemm_tile.cuh: the CUDA-core kernel's, chain for
// chain), so infinities and NaN give what they give there, for the CUDA-core
// kernel's price (4096 x 4096 x 256 383 us). Doing only the marked rows'
// entries so, a serial sum per thread, took 17 ms where one sample marked all
// rows, 0.7 ms for one NaN.
//
// What bounds it: six bf16 products per multiply-add; 4096 x 4096 x 256 is
// 51.5 GFLOP of MMA, 27 us at the measured bf16 rate, and 3.4 waves of tiles
// run as 4. Measured (GB300, inputs in L2): 4096 x 4096 x 250 44 us (the
// CUDA-core kernel 381), 4096 x 9216 x 256 79 us (831), 4096 x 4096 x 1024
// 135 us (1466), 1000 x 4096 x 256 18 us (110), 4096 x 4096 x 32 23 us (55). The
// MMAs alone take 1.8 us per 64 columns and wave, with the operand loads and the
// reading back 1.9 to 2.0; a wave's stores, of which the next tile's first
// columns hide part, 2-3 us; the look at the marks 1 us per call. x1 y1 read
// after every 32 columns instead of 64: 53 us at 256 columns, 161 at 1024;
// before the small products instead of after them: 2 to 4 us more; eight
// reading warps with 128 sums each (spilling): 10%; arrivals with
// .release.cluster 17-24%.
#include "gemm_tile.cuh"
#include "split_bf16.cuh"
#include "tc_pair.cuh"

namespace csrt {

constexpr int kGsStageCols = 64;                       // per pipeline stage: rows of 128 bytes
static_assert(kGsStageCols == kSplitChunk, "a stage is a sum of x1 y1");
constexpr int kGsSlice = 128 * kGsStageCols * 2;       // one plane of 128 rows: 16 KB
constexpr int kGsStageBytes = 6 * kGsSlice;            // three planes of each operand
constexpr int kGsStages = 2;
constexpr int kGsEpiWarps = 16;                        // per TMEM lane quarter four, 64 columns each
constexpr int kGsEpiCols = 64;
constexpr int kGsProd = 4;                             // a warpgroup of producers (TMA, MMA, two idle)
constexpr int kGsThreads = 32 * (kGsProd + kGsEpiWarps);
// register split (ptxas gives the launch 640 x 96; it is found to hold the
// shares before it is used): the sums (64), a block read back (16) and
// addresses need more than 96 in the epilogue warps; with 32 instead of 64 the
// producers spill
constexpr int kGsProdRegs = 64, kGsEpiRegs = 104;
constexpr int kGsSplitRegs = 128 * kGsProdRegs + 32 * kGsEpiWarps * kGsEpiRegs;
static_assert(kGsSplitRegs <= kGsThreads * 96, "register split");
constexpr int kGsTile = 256;
constexpr int kGsStageOut = 32 * 16 * 4;               // a 32 x 16 block on its way out
constexpr int kGsSmem = kGsStages * kGsStageBytes + kGsEpiWarps * kGsStageOut + 1024 + 256;
static_assert(kGsSmem <= 232448, "shared memory per block");
constexpr uint32_t kGsIdesc = idesc_bf16(256, 256);

struct GsArgs {
    float *g;
    int32_t m, k, n;
    const float *dy, *x;             // the float32 operands
    const uint8_t *marks;            // [num_marks] blocks of eight rows
    int32_t num_marks;
    int32_t tiles_k, num_tiles;
    WsHeader *hdr;
};

// Planes of rows 0..m-1 of dY and 0..k-1 of X (one warp per row, eight
// columns per lane and step).
__global__ void __launch_bounds__(256) split_rows_kernel(const float *__restrict__ dy, const float *__restrict__ x,
                                                         int32_t m, int32_t k, int32_t n, int32_t ld,
                                                         __nv_bfloat16 *__restrict__ pdy,
                                                         __nv_bfloat16 *__restrict__ px, uint8_t *__restrict__ marks,
                                                         int vec) {
    pdl_enter();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the GEMM's set-up may begin
    const int lane = threadIdx.x & 31;
    int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int cols = r < (int64_t)m + k ? n : 0;   // (the last block may have warps to spare)
    const bool is_x = r >= m;
    if (is_x) r -= m;
    const int64_t rows = is_x ? k : m;
    const float *src = (is_x ? x : dy) + r * n;
    __nv_bfloat16 *dst = (is_x ? px : pdy) + r * ld;
    const int64_t plane = rows * ld;
    bool bad = false;
    for (int c = lane * 8; c < cols; c += 256) {
        float v[8];
        if (vec && c + 8 <= n) {
            const float4 a = ldg_f4(src + c), b = ldg_f4(src + c + 4);
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
            v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = c + e < n ? __ldg(src + c + e) : 0.f;
        }
        __nv_bfloat162 p[3][4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            const float2 a = make_float2(v[e], v[e + 1]);
            if (!split_fits(a.x) || !split_fits(a.y)) bad = true;
            split_bf16(a, p[0][e / 2], p[1][e / 2], p[2][e / 2]);
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) *reinterpret_cast<uint4 *>(dst + q * plane + c) = *reinterpret_cast<uint4 *>(p[q]);
    }
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) marks[blockIdx.x] = bad;
}

// G by float32 multiply-adds, two 64 x 64 tiles at a time per CTA.
static __device__ __noinline__ void gs_plain(const GsArgs &a, uint8_t *smem) {
    const int group = threadIdx.x >> 8;
    if (group >= 2) return;
    GemmTileSmem &s = reinterpret_cast<GemmTileSmem *>(smem)[group];
    const int64_t tiles_k = (a.k + kGBN - 1) / kGBN, tiles = (int64_t)((a.m + kGBM - 1) / kGBM) * tiles_k;
    for (int64_t t = (int64_t)blockIdx.x * 2 + group; t < tiles; t += (int64_t)gridDim.x * 2)
        gemm_nt_tile(a.dy, a.x, a.m, a.k, a.n, 0, a.n, t / tiles_k * kGBM, t % tiles_k * kGBN, threadIdx.x & 255, s, a.g, 0,
                     [&] { asm volatile("bar.sync %0, 256;" ::"r"(1 + group) : "memory"); });
}

__global__ void __launch_bounds__(kGsThreads, 1)
    gemm_split_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, GsArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    float *epi = reinterpret_cast<float *>(smem + kGsStages * kGsStageBytes);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kGsStages * kGsStageBytes + kGsEpiWarps * kGsStageOut);
    uint64_t *empty = full + kGsStages;
    uint64_t *accf = empty + kGsStages;   // [2] the accumulator of x1 y1, that of the small products: ready
    uint64_t *acce = accf + 2;            // [2] read back (the leader's: all warps of both CTAs)
    uint64_t *fin = acce + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(fin + 1);
    __shared__ volatile int s_abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const int num_kb = (a.n + kGsStageCols - 1) / kGsStageCols;

    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < kGsStages; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accf + b, 1);
            mbar_init(acce + b, 2 * kGsEpiWarps);
        }
        mbar_init(fin, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_b)) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();   // the barriers of both CTAs are set up
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    // nothing before this reads or writes global memory: the set-up overlaps
    // the end of the split kernel, whose planes are complete from here on
    pdl_enter();
    bool marked = false;
    for (int i = threadIdx.x; i < a.num_marks; i += kGsThreads) marked |= a.marks[i] != 0;
    marked = __syncthreads_or(marked);   // the same for every CTA

    if (marked) {
        gs_plain(a, smem);
    } else if (warp < kGsProd) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kGsProdRegs));
    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            for (int t = pair; t < a.num_tiles && !s_abort; t += pairs) {
                const int m0 = (t / a.tiles_k) * kGsTile + (int)rank * 128;
                const int k0 = (t % a.tiles_k) * kGsTile + (int)rank * 128;
                for (int kb = 0; kb < num_kb; ++kb, ++it) {
                    const int s = it % kGsStages;
                    if (!pair_wait(empty + s, ((it / kGsStages) & 1) ^ 1, &s_abort)) break;
                    if (rank == 0) mbar_expect_tx(full + s, 2 * kGsStageBytes);
                    const uint32_t bar = map_to_rank(full + s, 0);
                    uint8_t *st = smem + s * kGsStageBytes;
#pragma unroll
                    for (int p = 0; p < 3; ++p) {
                        tma_load_2d_pair(st + p * kGsSlice, &map_a, kb * kGsStageCols, p * a.m + m0, bar);
                        tma_load_2d_pair(st + (3 + p) * kGsSlice, &map_b, kb * kGsStageCols, p * a.k + k0, bar);
                    }
                }
            }
            // every load of both CTAs must land before the pair may exit
            if (rank == 0)
                for (int i = imax(0, it - kGsStages); i < it; ++i)
                    mbar_wait(full + i % kGsStages, (i / kGsStages) & 1);
        }
    } else if (warp == 1) {
        if (rank == 0 && lane == 0) {
            int it = 0;
            uint32_t turn = 0;   // bits 0 and 1: parity of the two accumulators
            for (int t = pair; t < a.num_tiles && !s_abort; t += pairs) {
                for (int kb = 0; kb < num_kb; ++kb, ++it) {
                    const int s = it % kGsStages, in_flush = kb % kSplitFlush;
                    // steps of 16 columns (the last stage's columns past n are zero)
                    const int steps = imin(kGsStageCols, a.n - kb * kGsStageCols + 15) / 16;
                    if (!pair_wait(full + s, (it / kGsStages) & 1, &s_abort)) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t da = smem_desc_lo(smem + s * kGsStageBytes), db = da + (3 * kGsSlice >> 4);
                    if (in_flush == 0) {
                        if (!pair_wait(acce + 1, (turn >> 1) ^ 1, &s_abort)) break;
                        turn ^= 2;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    }
                    // the small products first (while they run, the sum of x1 y1
                    // before is read): parts of dY and of X by steps of four bits
#pragma unroll 1
                    for (int q = 0; q < 20; q += 4) {
                        const uint32_t qa = da + (kSplitPartsA >> q & 3) * (kGsSlice >> 4);
                        const uint32_t qb = db + (kSplitPartsB >> q & 3) * (kGsSlice >> 4);
#pragma unroll
                        for (int k = 0; k < kGsStageCols / 16; ++k)
                            if (k < steps) mma_bf16_pair(tmem + 256, qa + k * 2, qb + k * 2, kGsIdesc, k > 0 ? 1 : in_flush | q);
                    }
                    if (!pair_wait(acce, (turn & 1) ^ 1, &s_abort)) break;
                    turn ^= 1;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                    for (int k = 0; k < kGsStageCols / 16; ++k)
                        if (k < steps) mma_bf16_pair(tmem, da + k * 2, db + k * 2, kGsIdesc, k > 0);
                    mma_commit_pair(accf);
                    mma_commit_pair(empty + s);
                    if (in_flush == kSplitFlush - 1 || kb == num_kb - 1) mma_commit_pair(accf + 1);
                }
            }
            asm volatile(
                "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(fin))
                : "memory");
            mbar_wait(fin, 0);   // nothing of ours still runs on the tensor cores
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kGsEpiRegs));
        const int q = warp & 3;                  // TMEM lanes 32q ..: rows 32q .. of this CTA's 128
        const int h = (warp - kGsProd) >> 2;     // column quarter of the tile
        const uint32_t acce0 = map_to_rank(acce, 0), acce1 = map_to_rank(acce + 1, 0);
        float *xb = epi + (warp - kGsProd) * (kGsStageOut / 4);
        int sums = 0, flushes = 0;
        for (int t = pair; t < a.num_tiles; t += pairs) {
            const int64_t row = (int64_t)(t / a.tiles_k) * kGsTile + rank * 128 + q * 32 + lane;
            const int64_t col0 = (int64_t)(t % a.tiles_k) * kGsTile + h * kGsEpiCols;
            float acc[kGsEpiCols];
#pragma unroll
            for (int c = 0; c < kGsEpiCols; ++c) acc[c] = 0.f;
            bool ok = true;
            // (b = 0: the accumulator of x1 y1; 1: that of the small products)
            auto add_up = [&](int b, int times) {
                ok = __all_sync(0xffffffffu, pair_wait(accf + b, times & 1, &s_abort));
                if (!ok) return;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int c = 0; c < kGsEpiCols; c += 16) {
                    uint32_t r[16];
                    tmem_ld_16cols(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * 256 + h * kGsEpiCols + c), r);
#pragma unroll
                    for (int e = 0; e < 16; ++e) acc[c + e] += __uint_as_float(r[e]);
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(b ? acce1 : acce0);
            };
            for (int i = 1; i <= num_kb && ok; ++i) {
                add_up(0, sums++);
                if (ok && (i % kSplitFlush == 0 || i == num_kb)) add_up(1, flushes++);
            }
#pragma unroll
            for (int c = 0; c < kGsEpiCols; ++c) acc[c] *= kSplitDown;
            if (!ok) break;
            if (a.k % 8 == 0 && (reinterpret_cast<uintptr_t>(a.g) & 31) == 0) {
                // lane = row holds 64 columns; groups of four lanes exchange
                // 32-byte units so that lane j of a group holds unit j of each
                // of the group's rows: a store then covers eight whole lines
                // instead of a sector of 32 (4096 x 4096 x 32 27 -> 25 us)
                const int j = lane & 3;
#pragma unroll
                for (int c = 0; c < kGsEpiCols; c += 32) {
#pragma unroll
                    for (int sft = 1; sft <= 2; sft <<= 1) {
                        const bool up = (j & sft) != 0;
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            if (p & sft) continue;
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                float &lo = acc[c + p * 8 + e], &hi = acc[c + (p | sft) * 8 + e];
                                const float got = __shfl_xor_sync(0xffffffffu, up ? lo : hi, sft);
                                if (up) lo = got;
                                else hi = got;
                            }
                        }
                    }
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const int64_t r = row - j + p, col = col0 + c + j * 8;
                        if (r < a.m && col < a.k) st_global_f8(a.g + r * a.k + col, acc + c + p * 8);
                    }
                }
            } else {
                // any alignment: 32 x 16 blocks through shared memory, two
                // rows per store (16-byte chunk i of row r at i ^ ((r >> 1) & 3))
#pragma unroll
                for (int c = 0; c < kGsEpiCols; c += 16) {
                    __syncwarp();
#pragma unroll
                    for (int e = 0; e < 16; e += 4)
                        *reinterpret_cast<float4 *>(xb + lane * 16 + (e ^ (((lane >> 1) & 3) << 2))) =
                            make_float4(acc[c + e], acc[c + e + 1], acc[c + e + 2], acc[c + e + 3]);
                    __syncwarp();
                    const int cc = lane & 15;
                    const int64_t col = col0 + c + cc;
                    const int64_t rb = row - lane + (lane >> 4);
#pragma unroll 4
                    for (int i = 0; i < 32; i += 2) {
                        const int r = i + (lane >> 4);
                        if (rb + i < a.m && col < a.k) a.g[(rb + i) * a.k + col] = xb[r * 16 + (cc ^ (((r >> 1) & 3) << 2))];
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && s_abort) {
        dev_flag(a.hdr, CSRT_DEV_TIMEOUT);
        a.hdr->timeout_site = 11;
    }
    cluster_sync_all();   // no CTA leaves while the other may still use its shared memory
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

static int64_t gs_ld(int32_t n) { return ceil_div<int64_t>(n, 8) * 8; }
static size_t gs_align(size_t v) { return (v + 255) / 256 * 256; }

// Scratch of an m x k gradient over n columns: the planes and the marks.
static size_t gs_bytes(int64_t m, int64_t k, int32_t n) {
    return gs_align((size_t)(6 * m * gs_ld(n))) + gs_align((size_t)(6 * k * gs_ld(n))) +
           gs_align((size_t)ceil_div<int64_t>(m + k, 8)) + 256;
}

size_t gemm_split_scratch_bytes(int32_t rows, int32_t cols, int32_t max_n) {
    if (rows < 64 || cols < 64) return 0;
    const size_t cap = max_n <= 16384 ? (size_t)256 << 20 : (size_t)64 << 20;
    return imin(gs_bytes(rows, cols, max_n), cap);
}

int gemm_split_f32(const float *dy, const float *x, int32_t m, int32_t k, int32_t n, float *g, void *ws,
                   size_t ws_bytes, cudaStream_t s, bool *handled) {
    *handled = false;
    // under 32 columns a chain of multiply-adds is as exact and its time is
    // launch latency either way
    if (m < 64 || k < 64 || n < 32 || !device_is_sm10x()) return CSRT_OK;
    if (ws == nullptr || ws_bytes < kWsReservedBytes + gs_bytes(m, k, n)) return CSRT_OK;
    const int tiles_k = (int)ceil_div<int64_t>(k, kGsTile);
    const int tiles = (int)ceil_div<int64_t>(m, kGsTile) * tiles_k;
    const int pairs = imin(tiles, imax(1, num_sms() / 2));
    // Where the CUDA-core kernel is still faster: small outputs, few columns.
    // Both times fitted to measurements on GB300 (microseconds; the split
    // GEMM's over 64..4096 x 64..9216 x 32..1024 is met or up to 19% above what
    // it takes, the CUDA-core kernel's, a latency per column or its 22 TFLOP/s,
    // within 15%).
    const double waves = (double)ceil_div(tiles, pairs), chunks = (double)ceil_div(n, 32);
    const double t_split = 9.5 + waves * (2.5 + 1.0 * chunks);
    const double t_fma = imax(2.6 + 0.1 * imin(n, 512), 2.0 * m * k * n / 22e6);
    if (t_split > t_fma) return CSRT_OK;
    const int32_t ld = (int32_t)gs_ld(n);
    char *p = ws_scratch(ws);
    p = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(p) + 255) & ~uintptr_t(255));
    __nv_bfloat16 *pdy = reinterpret_cast<__nv_bfloat16 *>(p);
    p += gs_align((size_t)6 * m * ld);
    __nv_bfloat16 *px = reinterpret_cast<__nv_bfloat16 *>(p);
    p += gs_align((size_t)6 * k * ld);
    uint8_t *marks = reinterpret_cast<uint8_t *>(p);
    const int32_t num_marks = (int32_t)ceil_div<int64_t>((int64_t)m + k, 8);
    CUtensorMap ma, mb;
    if (!make_map_bf16(&ma, pdy, (int64_t)3 * m, n, ld, 128) ||
        !make_map_bf16(&mb, px, (int64_t)3 * k, n, ld, 128))
        return CSRT_OK;
    static std::atomic<int> ready[64];
    if (!pair_kernel_ready(gemm_split_kernel, ready, kGsSmem, kGsThreads, kGsSplitRegs)) return CSRT_OK;
    GsArgs a;
    a.g = g;
    a.m = m;
    a.k = k;
    a.n = n;
    a.dy = dy;
    a.x = x;
    a.marks = marks;
    a.num_marks = num_marks;
    a.tiles_k = tiles_k;
    a.num_tiles = tiles;
    a.hdr = static_cast<WsHeader *>(ws);
    const int vec = n % 4 == 0 && ((reinterpret_cast<uintptr_t>(dy) | reinterpret_cast<uintptr_t>(x)) & 15) == 0;
    launch_pdl(split_rows_kernel, dim3((unsigned)num_marks), dim3(256), 0, s, dy, x, m, k, n, ld, pdy, px, marks, vec);
    launch_pair(gemm_split_kernel, (unsigned)(2 * pairs), kGsThreads, kGsSmem, s, ma, mb, a);
    count_launch(2);
    *handled = true;
    return check_launch("gemm_split_kernel");
}

}  // namespace csrt
