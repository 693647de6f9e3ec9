// Sparse x dense products on the tensor cores: Y = W X for a CSR matrix dense
// enough that gathering a row of X per stored entry (n floats from L2 each)
// costs more than multiplying the zeros.
//
// The product runs as a GEMM over all of W's columns in float32 accuracy: both
// factors as sums of three bf16 parts, all 24 bits of every value and all of
// float32's exponents below 2^28, six of the nine products of parts, x1 w1 in
// sums of 64 columns that are added up with round to nearest (split_bf16.cuh).
// An element of Y thus has no part in the magnitudes of its neighbours: two
// fp16 parts, with a power of two per row of W and per 64 features x 64 columns
// of X, took half the products, but a sample 1e-16 times as large as another of
// its block was lost (relative error 0.2), W times unit vectors did not return
// W, and a sum of one term had up to 5.1e-7 where float32's rounding is 6e-8.
// Measured error against 64 bits: 0.7e-7 to 1.6e-7 where the float32 chain of the
// sparse kernel has 1.7e-7 to 7.8e-7 (rows of 120 to 2000 entries); layers whose
// rows hold fewer than 160 entries on average keep the sparse kernel.
//
// W exists in no other form than its CSR arrays: the first kernel (spmm_tc.cuh)
// notes where each row's 64-column chunks begin (4 bytes per row and chunk),
// and eight warps of each CTA put a chunk's entries into the cleared
// shared-memory operand of the MMA. (Copies of the entries, sorted by 16 rows and
// 64 columns, 6 bytes per entry of the capacity, took the workspace of a
// 4096 x 9216 layer at 256 columns from 52 to 276 MB; they were faster only
// where several column tiles each expand a very dense W, 4096 x 4096 x 1024 at
// 50% 223 against 278 us, and slower else, x 256 at 20% 70 against 65.)
//
// Work: (256-row tile, kN columns of X) x 64-column chunks, cut into one
// contiguous range per CTA pair. A pair whose range covers part of a tile's
// chunks leaves a partial sum; the tile's pairs then share its columns and
// add the parts up in pair order (st_share). Where there are enough tiles for
// the GPU no tile is cut.
//
// Measured (GB300; the sparse kernel's time in brackets), rows x inner x n:
// 4096 x 4096 x 256 at 20% 65 us (160), at 50% 104 (387), x 1024 at 5% 142
// (169), at 50% 278 (1530); 4096 x 9216 x 256 at 5% 87 (98), at 20% 122 (365).
// The MMAs take 1.7 us per chunk (six products; 24 of K = 16), with the
// operands and the reading back 1.9. From about 15% the expanding warps bound
// it (4096 x 4096 x 1024 at 50%: 3.9 us per chunk; without the entries past each
// row's sixteenth 182 us in all): some 700 instructions per warp and chunk, one
// at a time. More of them in flight did not help: four rounds asked for ahead,
// which took registers from the warps that add up, 268 us at 50% and 154
// instead of 143 at 5%. The first kernel takes 40 us at 50%, the partial sums
// of cut tiles 7 (20 MB written and read in L2).
//
// Operands that the tensor cores can't take (values of 2^28 and more, infinities,
// NaN, rows out of order or with an entry twice) are marked by the first kernel
// and make the whole product run by gathering (st_gather).
#include "spmm_tc.cuh"
#include "tc_pair.cuh"

namespace csrt {

constexpr int kStChunk = kTcChunk;
static_assert(kStChunk == kSplitChunk, "a stage is a sum of x1 w1");
// Warps: 0 TMA, 1 MMA (2 and 3 idle), eight that expand W (a group of 16 rows
// each), sixteen that add up and write. kStSplitRegs: what their shares come to
// (the launch is found to hold them before it is used; ptxas gives 896 x 72).
constexpr int kStExpandWarps = 8, kStEpiWarps = 16;
constexpr int kStThreads = 32 * (4 + kStExpandWarps + kStEpiWarps);
constexpr int kStProdRegs = 32, kStExpandRegs = 40, kStEpiRegs = 96;
constexpr int kStSplitRegs =
    128 * kStProdRegs + 32 * (kStExpandWarps * kStExpandRegs + kStEpiWarps * kStEpiRegs);
static_assert(kStSplitRegs <= kStThreads * 72, "register split");
constexpr int kStASlice = 128 * kStChunk * 2;
template <int kN> __host__ __device__ constexpr int st_bslice() { return kN / 2 * kStChunk * 2; }
template <int kN> __host__ __device__ constexpr int st_stage() { return 3 * (kStASlice + st_bslice<kN>()); }
template <int kN> __host__ __device__ constexpr int st_stages() { return kN == 256 ? 2 : 3; }
template <int kN> __host__ __device__ constexpr int st_smem() { return st_stages<kN>() * st_stage<kN>() + 256 + 1024; }
static_assert(st_smem<256>() <= 232448 && st_smem<128>() <= 232448, "shared memory per block");

struct StArgs {
    const int32_t *row_ptr, *col;
    const float *val;
    int32_t rows, k, n;
    const int32_t *start;
    const float *x;
    float *y, *partial;
    uint32_t *cnt;
    const uint8_t *marks;
    int32_t num_marks;
    const float *bias, *mask;
    int32_t relu;
    int64_t nnz_min;
    int32_t tiles_n, tiles, chunks, pairs;
    int32_t whole;   // pairs take whole tiles
    int32_t vec;     // rows of X may be read as float4
    WsHeader *hdr;
};

__device__ __forceinline__ int32_t ld_row_end(const int32_t *p) {
    int32_t v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ float st_finish(const StArgs &a, int64_t row, int64_t c, float v) {
    if (a.bias) v = __fadd_rn(v, __ldg(a.bias + row));
    if (a.relu) v = fmaxf(v, 0.f);
    if (a.mask && !(__ldg(a.mask + row * a.n + c) > 0.f)) v = 0.f;
    return v;
}

// The whole product by gathering, for operands that the tensor cores can't take
// (marked by the first kernel): a warp per row and 32 VW columns, which lie VW
// to a lane; the row's entries in their order, one chain of multiply-adds per
// element of Y.
template <int VW>
static __device__ __noinline__ void st_gather(const StArgs &a) {
    const int lane = threadIdx.x & 31;
    const int tiles = (a.n + 32 * VW - 1) / (32 * VW);
    const int64_t work = (int64_t)a.rows * tiles, step = (int64_t)gridDim.x * (kStThreads / 32);
    for (int64_t i = (int64_t)blockIdx.x * (kStThreads / 32) + (threadIdx.x >> 5); i < work; i += step) {
        const int64_t row = i / tiles;
        const int c = (int)(i % tiles) * 32 * VW + lane * VW;   // (a multiple of VW in n: all of a lane's or none)
        const bool on = c < a.n;
        float sum[VW] = {};
        const int32_t end = __ldg(a.row_ptr + row + 1);
        for (int32_t e0 = __ldg(a.row_ptr + row); e0 < end; e0 += 32) {
            const int32_t cnt = min(32, end - e0);
            const int32_t col = lane < cnt ? __ldg(a.col + e0 + lane) : 0;
            const float val = lane < cnt ? __ldg(a.val + e0 + lane) : 0.f;
            for (int e = 0; e < cnt; e += 8) {
                float x[8][VW];
#pragma unroll
                for (int o = 0; o < 8; ++o) {   // eight rows of X in flight
                    const int64_t j = __shfl_sync(0xffffffffu, col, e + o);
                    const float *p = a.x + j * a.n + c;
                    if (e + o >= cnt || !on) continue;
                    if constexpr (VW == 4) {
                        const float4 v = ldg_f4(p);
                        x[o][0] = v.x; x[o][1] = v.y; x[o][2] = v.z; x[o][3] = v.w;
                    } else {
                        x[o][0] = __ldg(p);
                    }
                }
#pragma unroll
                for (int o = 0; o < 8; ++o) {
                    const float w = __shfl_sync(0xffffffffu, val, e + o);
                    if (e + o >= cnt || !on) continue;
#pragma unroll
                    for (int v = 0; v < VW; ++v) sum[v] = fmaf(w, x[o][v], sum[v]);
                }
            }
        }
        if (!on) continue;
#pragma unroll
        for (int v = 0; v < VW; ++v) a.y[row * a.n + c + v] = st_finish(a, row, c + v, sum[v]);
    }
}

// First unit of pair p, and the pair that unit u belongs to.
__host__ __device__ inline int64_t st_first(int64_t units, int pairs, int p) { return units * p / pairs; }
__host__ __device__ inline int st_pair_of(int64_t units, int pairs, int64_t u) {
    return (int)(((u + 1) * pairs - 1) / units);
}
// The partial sum a pair leaves of a tile it shares: two slots per pair (the
// beginning of a tile, or a later part) and CTA, 128 x kN floats each.
template <int kN>
__device__ __forceinline__ float *st_slot(const StArgs &a, int pair, bool beginning, uint32_t rank) {
    return a.partial + ((int64_t)(pair * 2 + (beginning ? 1 : 0)) * 2 + rank) * 128 * kN;
}

// Eight columns (c .. c + 7 of the tile) of row 32q + lane of the CTA's half
// of a tile: the sums without the factors' scales, the epilogue, Y.
template <int kN>
__device__ __forceinline__ void st_write(const StArgs &a, int tile, uint32_t rank, int q, int c,
                                         const float *sum) {
    const int64_t row = (int64_t)(tile / a.tiles_n) * 256 + rank * 128 + q * 32 + (threadIdx.x & 31);
    const int64_t col = (int64_t)(tile % a.tiles_n) * kN + c;
    if (row >= a.rows || col >= a.n) return;
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = sum[i] * kSplitDown;
    if (a.bias || a.relu || a.mask) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (col + i < a.n) v[i] = st_finish(a, row, col + i, v[i]);
    }
    float *dst = a.y + row * a.n + col;
    if (a.n % 8 == 0 && (reinterpret_cast<uintptr_t>(a.y) & 31) == 0) {
        st_global_f8(dst, v);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (col + i < a.n) dst[i] = v[i];
    }
}

// Counting in at a cut tile: the parts that are there (bits 0-7) and the
// shares whose pairs gave up waiting (from bit 8). The first kernel of every
// product zeroes the counters.
constexpr uint32_t kStPartsMask = 0xff;
// How long a pair waits for the others' parts: 15 us at 2 GHz, or this many
// looks (each a round trip to L2, up to 1 to 2 us under the load of the
// partial sums: by their number alone the wait could last 25 times as long).
constexpr long long kStShareClocks = 30000;
constexpr int kStSharePolls = 400;

// One pair's part in adding up a cut tile; `seen` is what its counter was when
// it counted in.
template <int kN>
__device__ __noinline__ void st_share(const StArgs &a, int64_t units, int pair, int tile, uint32_t rank, int q, int h,
                                      int tid, uint32_t seen, volatile uint32_t *state) {
    constexpr int kUnits = kN / 32;   // eights of an epilogue warp's columns
    const int64_t t0 = (int64_t)tile * a.chunks;
    const int p0 = st_pair_of(units, a.pairs, t0), parts = st_pair_of(units, a.pairs, t0 + a.chunks - 1) - p0 + 1;
    // (the pair that begins a tile has ended another, whose share it does)
    const int shares = imin(parts - 1, kUnits), own = pair - p0 - 1;
    uint32_t *cnt = a.cnt + (tile * 2 + (int)rank);
    if (tid == 0) {
        uint32_t todo = own >= 0 && own < shares ? 1u << own : 0u;
        if ((int)(seen & kStPartsMask) == parts - 1) {
            todo |= seen >> 8;   // the last to come: also the shares given up before
            __threadfence();
        } else if (todo) {
            bool all = false;
            const long long begun = clock64();
            for (int i = 0; i < kStSharePolls; ++i) {
                uint32_t now;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(cnt) : "memory");
                if ((all = (int)(now & kStPartsMask) == parts) || clock64() - begun > kStShareClocks) break;
                __nanosleep(20);
            }
            // gives up; whoever counts in last takes the share, unless it just has
            if (!all && (int)(atomicOr(cnt, todo << 8) & kStPartsMask) != parts) todo = 0;
            if (!all) __threadfence();
        }
        *state = todo;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kStEpiWarps) : "memory");
    uint32_t todo = *state;
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kStEpiWarps) : "memory");   // state is read
    for (; todo; todo &= todo - 1) {
        const int s = __ffs((int)todo) - 1;
        for (int c = kUnits * s / shares; c < kUnits * (s + 1) / shares; ++c) {
            // six parts' loads in flight (a tile rarely has more): the time here
            // is that of the L2 round trips, 1 to 2 us each under this load
            float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            for (int p = 0; p < parts; p += 6) {
                float x[6][8];
#pragma unroll
                for (int o = 0; o < 6; ++o)
                    if (p + o < parts)
                        ld_global_f8(st_slot<kN>(a, p0 + p + o, p + o == 0, rank) + (c * 32 * kStEpiWarps + tid) * 8, x[o]);
#pragma unroll
                for (int o = 0; o < 6; ++o)
                    if (p + o < parts) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] += x[o][i];
                    }
            }
            st_write<kN>(a, tile, rank, q, h * (kN / 4) + c * 8, v);
        }
    }
}

template <int kN>
__global__ void __launch_bounds__(kStThreads, 1)
    spmm_tc_kernel(const __grid_constant__ CUtensorMap map_x, StArgs a) {
    // The first kernel's blocks have all passed their own wait when this kernel
    // starts, so the row pointers (which it does not write) are complete.
    if (ld_row_end(a.row_ptr + a.rows) < a.nnz_min) {
        pdl_enter();   // (whoever waits for this kernel waits for the one before, too)
        return;        // the sparse kernel before this one does the product
    }
    constexpr int kStages = st_stages<kN>(), kStage = st_stage<kN>(), kBSlice = st_bslice<kN>();
    constexpr int kCols = kN / 4;   // columns of an epilogue warp
    constexpr uint32_t kIdesc = idesc_bf16(256, kN);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kStages * kStage);
    uint64_t *empty = full + kStages;
    uint64_t *accf = empty + kStages;   // [2] the accumulator of x1 w1, that of the small products: ready
    uint64_t *acce = accf + 2;          // [2] read (the leader's: all warps of both CTAs)
    uint64_t *fin = acce + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(fin + 1);
    __shared__ volatile int s_abort;
    __shared__ volatile uint32_t s_state;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1;
    const int64_t units = (int64_t)a.tiles * a.chunks;
    const int64_t u_begin = a.whole ? st_first(a.tiles, a.pairs, pair) * a.chunks : st_first(units, a.pairs, pair);
    const int64_t u_end = a.whole ? st_first(a.tiles, a.pairs, pair + 1) * a.chunks : st_first(units, a.pairs, pair + 1);

    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full + s, 1 + 2 * kStExpandWarps);
            mbar_init(empty + s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accf + b, 1);
            mbar_init(acce + b, 2 * kStEpiWarps);
        }
        mbar_init(fin, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_x)) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(2 * kN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    pdl_enter();   // the operands are complete from here on
    bool marked = false;
    for (int i = threadIdx.x; i < a.num_marks; i += kStThreads) marked |= a.marks[i] != 0;
    marked = __syncthreads_or(marked);   // the same for every CTA

    if (marked) {
        if (a.vec) st_gather<4>(a);
        else st_gather<1>(a);
    } else if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kStProdRegs));
        // (few registers here: what changes is the stage, its barriers' parity, and
        // those of the accumulators)
        const int stages = (int)(u_end - u_begin);
        int ch = (int)(u_begin % a.chunks), st = 0;
        uint32_t turn = 0;   // bit 0: parity of the stages' round; 1, 2: of the accumulators
        if (warp == 0 && lane == 0) {
            int c0 = (int)(u_begin / a.chunks % a.tiles_n) * kN + (int)rank * (kN / 2);
            int done = 0;
            for (; done < stages && !s_abort; ++done) {
                if (!pair_wait(empty + st, (turn & 1) ^ 1, &s_abort)) break;
                if (rank == 0) mbar_expect_tx(full + st, 6 * kBSlice);
                const uint32_t bar = map_to_rank(full + st, 0);
                uint8_t *to = smem + st * kStage + 3 * kStASlice;
#pragma unroll
                for (int p = 0; p < 3; ++p)
                    tma_load_2d_pair(to + p * kBSlice, &map_x, ch * kStChunk, p * a.n + c0, bar);
                if (++ch == a.chunks) {
                    ch = 0;
                    c0 += kN;
                    if (c0 >= a.tiles_n * kN) c0 = (int)rank * (kN / 2);
                }
                if (++st == kStages) st = 0, turn ^= 1;
            }
            // every load of both CTAs must land before the pair may exit
            if (rank == 0)
                for (int i = imax(0, done - kStages); i < done; ++i) mbar_wait(full + i % kStages, (i / kStages) & 1);
        } else if (warp == 1 && lane == 0 && rank == 0) {
            int in_flush = 0;
            for (int done = 1; done <= stages && !s_abort; ++done) {
                if (!pair_wait(full + st, turn & 1, &s_abort)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // (a descriptor's low bits are the address in units of 16 bytes)
                const uint32_t da = smem_desc_lo(smem + st * kStage);
                if (in_flush == 0) {
                    if (!pair_wait(acce + 1, (turn >> 2) ^ 1, &s_abort)) break;
                    turn ^= 4;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                }
                // the small products first (while they run, the sum of x1 w1 before
                // is read): parts of W and of X by steps of four bits
#pragma unroll 1
                for (int q = 0; q < 20; q += 4) {
                    const uint32_t qa = da + (kSplitPartsA >> q & 3) * (kStASlice >> 4);
                    const uint32_t qb = da + (3 * kStASlice >> 4) + (kSplitPartsB >> q & 3) * (kBSlice >> 4);
#pragma unroll
                    for (int k = 0; k < kStChunk / 16; ++k)
                        mma_bf16_pair(tmem + kN, qa + k * 2, qb + k * 2, kIdesc, k > 0 ? 1 : in_flush | q);
                }
                if (!pair_wait(acce, (turn >> 1 & 1) ^ 1, &s_abort)) break;
                turn ^= 2;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int k = 0; k < kStChunk / 16; ++k)
                    mma_bf16_pair(tmem, da + k * 2, da + (3 * kStASlice >> 4) + k * 2, kIdesc, k > 0);
                mma_commit_pair(accf);
                ++in_flush;
                mma_commit_pair(empty + st);
                if (++ch == a.chunks) ch = 0;
                if (in_flush == kSplitFlush || ch == 0 || done == stages) {
                    mma_commit_pair(accf + 1);
                    in_flush = 0;
                }
                if (++st == kStages) st = 0, turn ^= 1;
            }
            asm volatile(
                "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(fin))
                : "memory");
            mbar_wait(fin, 0);
        }
    } else if (warp < 4 + kStExpandWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kStExpandRegs));
        // An expanding warp: one group of 16 rows. Per chunk it clears their
        // 128 bytes in the three planes and puts the entries' parts at their
        // places: eight lanes to a row, four rows at a time, eight entries of
        // every row per round. Two rounds are asked for as soon as the chunk
        // before is in place, and the bounds of the rows' runs one chunk
        // earlier: their latency (1000 clocks under load) passes while the MMAs
        // of the stage ahead run.
        const int e = warp - 4;
        const int groups = (a.rows + kTcGroup - 1) / kTcGroup;
        const int sub = lane & 7, quad = lane >> 3;
        int tile = (int)(u_begin / a.chunks), ch = (int)(u_begin % a.chunks);
        // the next unit's bounds: lane r the first entry of row r, lane 16 + r its end
        int64_t asked = u_begin;
        auto next_bounds = [&]() -> int32_t {
            if (asked >= u_end) return 0;
            const int g = (tile / a.tiles_n) * 16 + (int)rank * 8 + e;
            const int32_t got = g < groups ? __ldg(a.start + ((int64_t)g * (a.chunks + 1) + ch) * kTcGroup + lane) : 0;
            ++asked;
            if (++ch == a.chunks) {
                ch = 0;
                ++tile;
            }
            return got;
        };
        int32_t col[2][4];
        float val[2][4];
        auto fetch = [&](int32_t bounds, int round) {
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int r = (s >> 1) * 8 + (s & 1) + quad * 2;
                const int32_t lo = __shfl_sync(0xffffffffu, bounds, r) + round * 8 + sub;
                const int32_t hi = __shfl_sync(0xffffffffu, bounds, 16 + r);
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const int32_t i = lo + o * 8;
                    col[o][s] = i < hi ? __ldg(a.col + i) : -1;
                    val[o][s] = i < hi ? __ldg(a.val + i) : 0.f;
                }
            }
        };
        // (column j of row r lies at r * 128 + (2 j ^ (r & 7) * 16): 128-byte swizzle)
        const uint32_t first = smem_u32(smem) + (uint32_t)(e * (kTcGroup * 128) + quad * 256);
        auto put = [&](uint32_t at0) {
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                __nv_bfloat162 part[3];
                split_bf16(make_float2(val[0][s], val[1][s]), part[0], part[1], part[2]);
                const uint32_t turn = (uint32_t)((s & 1) * 16 + quad * 32);
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const uint32_t at = at0 + (s >> 1) * 1024 + (s & 1) * 128 + (((uint32_t)col[o][s] * 2 & 126) ^ turn);
                    const uint32_t w1 = *reinterpret_cast<const uint32_t *>(&part[0]);
                    const uint32_t w2 = *reinterpret_cast<const uint32_t *>(&part[1]);
                    const uint32_t w3 = *reinterpret_cast<const uint32_t *>(&part[2]);
                    asm volatile(
                        "{\n .reg .pred p;\n setp.ge.s32 p, %4, 0;\n @p st.shared.u16 [%0], %1;\n"
                        " @p st.shared.u16 [%0 + %5], %2;\n @p st.shared.u16 [%0 + %6], %3;\n}\n" ::"r"(at),
                        "h"((uint16_t)(o ? w1 >> 16 : w1)), "h"((uint16_t)(o ? w2 >> 16 : w2)),
                        "h"((uint16_t)(o ? w3 >> 16 : w3)), "r"(col[o][s]), "n"(kStASlice), "n"(2 * kStASlice)
                        : "memory");
                }
            }
        };
        int32_t bounds = next_bounds(), bounds_n = next_bounds();
        fetch(bounds, 0);
        int it = 0;
        for (int64_t u = u_begin; u < u_end; ++u, ++it) {
            const int s = it % kStages;
            uint8_t *base = smem + s * kStage + e * (kTcGroup * 128);
            if (!__all_sync(0xffffffffu, pair_wait(empty + s, ((it / kStages) & 1) ^ 1, &s_abort))) break;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
                for (int p = 0; p < 3; ++p)
                    *reinterpret_cast<uint4 *>(base + p * kStASlice + i * 512 + lane * 16) = make_uint4(0, 0, 0, 0);
            }
            __syncwarp();
            put(first + s * kStage);
            const int run = __shfl_sync(0xffffffffu, bounds, 16 | lane) - bounds;   // (of lanes under 16)
            const int longest = __reduce_max_sync(0xffffffffu, lane < 16 ? run : 0);
            for (int round = 2; round * 8 < longest; round += 2) {
                fetch(bounds, round);
                put(first + s * kStage);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_to_rank(full + s, 0));
            bounds = bounds_n;
            fetch(bounds, 0);
            bounds_n = next_bounds();
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kStEpiRegs));
        const int q = warp & 3;             // TMEM lanes 32q ..
        const int h = (warp - 4 - kStExpandWarps) >> 2;   // column quarter of the tile
        const int tid = threadIdx.x - 32 * (4 + kStExpandWarps);
        const uint32_t acce0 = map_to_rank(acce, 0), acce1 = map_to_rank(acce + 1, 0);
        int sums = 0, flushes = 0, tile_e = -1, tile_b = -1;
        uint32_t seen_e = 0, seen_b = 0;   // (thread 0)
        bool ok = true;
        for (int64_t u = u_begin; u < u_end;) {
            const int tile = (int)(u / a.chunks), ch0 = (int)(u % a.chunks);
            const int ch1 = (int)imin<int64_t>(a.chunks, ch0 + (u_end - u));
            float acc[kCols];
#pragma unroll
            for (int c = 0; c < kCols; ++c) acc[c] = 0.f;
            // (b = 0: the accumulator of x1 w1; 1: that of the small products)
            auto add_up = [&](int b, int times) {
                ok = __all_sync(0xffffffffu, pair_wait(accf + b, times & 1, &s_abort));
                if (!ok) return;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int c = 0; c < kCols; c += 16) {
                    uint32_t r[16];
                    tmem_ld_16cols(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * kN + h * kCols + c), r);
#pragma unroll
                    for (int i = 0; i < 16; ++i) acc[c + i] += __uint_as_float(r[i]);
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(b ? acce1 : acce0);
            };
            const int sums_here = ch1 - ch0;
            for (int i = 1; i <= sums_here && ok; ++i) {
                add_up(0, sums++);
                if (ok && (i % kSplitFlush == 0 || i == sums_here)) add_up(1, flushes++);
            }
            if (!ok) break;
            u += ch1 - ch0;
            if (ch0 == 0 && ch1 == a.chunks) {
#pragma unroll
                for (int c = 0; c < kCols; c += 8) st_write<kN>(a, tile, rank, q, h * kCols + c, acc + c);
                continue;
            }
            // A partial sum: left in the workspace, counted in. (A pair's
            // first range may end a tile, its last may begin one.)
            const bool begins = ch0 == 0;
            float *mine = st_slot<kN>(a, pair, begins, rank) + tid * 8;
#pragma unroll
            for (int c = 0; c < kCols; c += 8) st_global_f8(mine + c * (32 * kStEpiWarps), acc + c);
            __threadfence();
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kStEpiWarps) : "memory");
            if (tid == 0) {
                const uint32_t seen = atomicAdd(a.cnt + (tile * 2 + (int)rank), 1u);
                if (begins) seen_b = seen;
                else seen_e = seen;
            }
            if (begins) tile_b = tile;
            else tile_e = tile;
        }
        // The cut tiles: their pairs share the work of adding the partial
        // sums (in pair order, so the result does not depend on who adds).
        // All pairs finish at about the same time: each waits a moment
        // (kStShareClocks) until a tile's parts are all there and takes its own
        // share of the columns. One that has waited in vain leaves a note and
        // goes; the last pair to count in does the shares of those, so
        // nothing depends on all pairs being resident at once.
        if (ok) {
            if (tile_e >= 0) st_share<kN>(a, units, pair, tile_e, rank, q, h, tid, seen_e, &s_state);
            if (tile_b >= 0) st_share<kN>(a, units, pair, tile_b, rank, q, h, tid, seen_b, &s_state);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && s_abort) {
        dev_flag(a.hdr, CSRT_DEV_TIMEOUT);
        a.hdr->timeout_site = 12;
    }
    cluster_sync_all();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kN) : "memory");
    }
}

static size_t st_align(size_t v) { return (v + 255) / 256 * 256; }
static int32_t st_ld(int32_t k) { return (int32_t)ceil_div<int64_t>(k, 8) * 8; }
static int st_max_pairs() { return imax(1, num_sms() / 2); }
// Row starts, planes, marks, counters and partial sums of a rows x k matrix and n
// columns.
static size_t st_bytes(int32_t rows, int32_t k, int32_t n, int n_tile) {
    const int64_t chunks = ceil_div(k, kStChunk);
    return st_align((size_t)6 * n * st_ld(k)) +
           st_align((size_t)4 * kTcGroup * ceil_div(rows, kTcGroup) * (chunks + 1)) +
           st_align((size_t)ceil_div(rows, kTcGroup) + chunks * ceil_div(n, n_tile / 4)) +
           st_align((size_t)8 * ceil_div(rows, 256) * ceil_div(n, n_tile)) + (size_t)st_max_pairs() * 4 * 128 * n_tile * sizeof(float) + 512;
}
constexpr int32_t kStMinRows = 256, kStMinK = 1024, kStMinN = 65;
constexpr int32_t kStMaxTiles = 4096;
static bool st_shape_ok(int32_t rows, int32_t k) {
    return rows >= kStMinRows && k >= kStMinK && k <= kTcMaxChunks * kStChunk;
}

size_t spmm_tc_scratch_bytes(int32_t rows, int32_t cols, int32_t max_n) {
    if (max_n < kStMinN) return 0;
    const bool fwd = st_shape_ok(rows, cols), bwd = st_shape_ok(cols, rows);
    if (!fwd && !bwd) return 0;
    const size_t f = fwd ? st_bytes(rows, cols, max_n, 256) : 0, b = bwd ? st_bytes(cols, rows, max_n, 256) : 0;
    return imax(f, b) <= (size_t)1 << 30 ? imax(f, b) : 0;   // beyond a gigabyte: the sparse kernel alone
}

void spmm_tc_plan(int32_t rows, int32_t k, int32_t n, int64_t capacity, const float *x, void *ws, size_t ws_bytes,
                  int32_t sparse_units, double t_entry, SpmmTcPlan *plan) {
    plan->prep.nnz_min = 0;
    if (!st_shape_ok(rows, k) || n < kStMinN || ws == nullptr || !device_is_sm10x()) return;
    const int n_tile = n <= 128 ? 128 : 256;
    capacity = imin<int64_t>(capacity, (int64_t)rows * k);
    if (ws_bytes < kWsReservedBytes + st_bytes(rows, k, n, n_tile)) return;
    const int chunks = ceil_div(k, kStChunk);
    plan->n_tile = n_tile;
    plan->tiles_n = ceil_div(n, n_tile);
    if ((int64_t)ceil_div(rows, 256) * plan->tiles_n > kStMaxTiles) return;
    plan->tiles = ceil_div(rows, 256) * plan->tiles_n;
    const int64_t units = (int64_t)plan->tiles * chunks;
    // Whole tiles per pair where that costs no more than cutting them
    // (microseconds; the partial sums take 4 us and 2.2 us for each eighth of
    // a tile's columns that a pair has to add up).
    const int max_pairs = st_max_pairs();
    const double t_unit = n_tile == 256 ? 1.85 : 1.75;
    const int cut_pairs = (int)imin<int64_t>(units, max_pairs);
    const double whole = (double)ceil_div(plan->tiles, max_pairs) * chunks * t_unit;
    const double cut = (double)ceil_div<int64_t>(units, cut_pairs) * t_unit + 4.0 +
                       2.2 * ceil_div(n_tile / 32, imax(1, cut_pairs / plan->tiles));
    plan->whole = whole <= cut;
    plan->pairs = plan->whole ? ceil_div(plan->tiles, ceil_div(plan->tiles, max_pairs)) : cut_pairs;
    // The number of entries from which this path is the faster one: both
    // times are fits to measurements over 512..9216 rows and columns, 3% to
    // 20% and 99 to 1024 columns of X (within 8%):
    //   here    14 us (both operands, launches, first and last steps), the
    //           chunks, 4e-6 us per entry (until the expanding warps bound it,
    //           from about 15%);
    //   sparse  8.5 us and t_entry per entry.
    // Where the two meet, 0.95 of what they give is what was measured: 4096 x
    // 4096 x 256 5.5%, x 1024 4.1%, 4096 x 9216 x 256 4.4% (at 5% 87 us against
    // 98), 1300 x 5000 x 99 5.6%.
    // And the number from which it is the more exact one: a sum of the sparse
    // kernel runs over a row, or over the part of it in one unit, and its
    // error grows with that length (1.0e-7 at 50, 1.4e-7 at 110, 1.7e-7 at
    // 120 to 200, 7.8e-7 at 2000), here it is 0.7e-7 to 1.6e-7.
    const double t_tc = 14.0 + imin(whole, cut);
    if (t_entry <= 5e-6) return;
    const int64_t nnz_min = imax<int64_t>(imax<int64_t>((int64_t)rows * 160, (int64_t)sparse_units * 128),
                                          (int64_t)(0.95 * (t_tc - 8.5) / (t_entry - 4e-6)));
    // Where the sparse kernel turns out to be the better one, the launch that
    // follows it in vain costs 1.5 us (and the host 4): not where only the
    // densest matrices would gain.
    if (nnz_min > capacity || (double)nnz_min > 0.09 * rows * k) return;
    char *p = ws_scratch(ws);
    p = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(p) + 255) & ~uintptr_t(255));
    auto take = [&](size_t bytes) {
        char *at = p;
        p += st_align(bytes);
        return at;
    };
    plan->prep.xp = reinterpret_cast<__nv_bfloat16 *>(take((size_t)6 * n * st_ld(k)));
    plan->prep.start = reinterpret_cast<int32_t *>(take((size_t)4 * kTcGroup * ceil_div(rows, kTcGroup) * (chunks + 1)));
    plan->prep.num_marks = ceil_div(rows, kTcGroup) + chunks * ceil_div(n, n_tile / 4);
    plan->prep.marks = reinterpret_cast<uint8_t *>(take((size_t)plan->prep.num_marks));
    plan->prep.counters = 2 * plan->tiles;
    plan->prep.cnt = reinterpret_cast<uint32_t *>(take((size_t)4 * plan->prep.counters));
    plan->partial = reinterpret_cast<float *>(p);
    plan->prep.k = k;
    plan->prep.ld = st_ld(k);
    plan->prep.chunks = chunks;
    plan->prep.width = n_tile / 4;
    plan->prep.vec = n % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
    if (!make_map_bf16(&plan->map_x, plan->prep.xp, (int64_t)3 * n, k, plan->prep.ld, n_tile / 2)) return;
    static std::atomic<int> ready256[64], ready128[64];
    if (!(n_tile == 256 ? pair_kernel_ready(spmm_tc_kernel<256>, ready256, st_smem<256>(), kStThreads, kStSplitRegs)
                        : pair_kernel_ready(spmm_tc_kernel<128>, ready128, st_smem<128>(), kStThreads, kStSplitRegs)))
        return;
    plan->prep.nnz_min = nnz_min;
}

int spmm_tc_launch(const SpmmTcPlan &plan, const int32_t *row_ptr, const int32_t *col, const float *val, int32_t rows,
                   const float *x, int32_t n, float *y, const float *bias, int32_t relu, const float *mask, void *ws,
                   cudaStream_t s) {
    StArgs a;
    a.row_ptr = row_ptr;
    a.col = col;
    a.val = val;
    a.rows = rows;
    a.k = plan.prep.k;
    a.n = n;
    a.start = plan.prep.start;
    a.x = x;
    a.y = y;
    a.partial = plan.partial;
    a.cnt = plan.prep.cnt;
    a.marks = plan.prep.marks;
    a.num_marks = plan.prep.num_marks;
    a.vec = plan.prep.vec;
    a.bias = bias;
    a.mask = mask;
    a.relu = relu;
    a.nnz_min = plan.prep.nnz_min;
    a.tiles_n = plan.tiles_n;
    a.tiles = plan.tiles;
    a.chunks = plan.prep.chunks;
    a.pairs = plan.pairs;
    a.whole = plan.whole;
    a.hdr = static_cast<WsHeader *>(ws);
    const unsigned grid = (unsigned)(2 * plan.pairs);
    if (plan.n_tile == 256) launch_pair(spmm_tc_kernel<256>, grid, kStThreads, st_smem<256>(), s, plan.map_x, a);
    else launch_pair(spmm_tc_kernel<128>, grid, kStThreads, st_smem<128>(), s, plan.map_x, a);
    count_launch();
    return check_launch("spmm_tc_kernel");
}

}  // namespace csrt
