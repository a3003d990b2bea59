// IF4 matrix product on the Blackwell tensor cores (tcgen05): C = A B^T for two IF4 (or NVFP4) operands with the
// arithmetic of the paper's MAC unit (Sec. 5.2): inside a pair of groups the decoded codes are multiplied and
// summed exactly, the sum is scaled by Delta_a * Delta_b, and the factors 1, 6/7 or 36/49 -- none, one or both
// groups stored as integers -- are applied in FP32 on the scale path, here in the epilogue.
//
// How integer groups reach an FP4 tensor core.  An FP4 group is an NVFP4 group (Sec. 3) and goes to
// tcgen05.mma kind::mxf4nvf4 as it is.  An integer code k in -8..7 stands for (6/7) k, which is no E2M1 value, but it is
// h + l / 7 with two of them: for |k| = 1, 2, 3, 4, 6 take h = k, l = -k (k - k/7 = 6k/7); for 5, 7 and 8 take
// (4, 2), (6, 0) and (6, 6).  So every operand is split once into two NVFP4 "planes" that share the group scales:
//     H: the codes of the FP groups, h of the integer groups     L: zero in the FP groups, l of the integer groups
// and the product is  H_a H_b  +  1/7 (H_a L_b + L_a H_b)  +  1/49 L_a L_b,  four block-scaled MMAs per K-step (an earlier
// split of k itself into two summands, beside a plane of the FP groups, took nine) into three FP32 accumulators that live
// in tensor memory side by side (3 x 128 columns) and meet only in the epilogue.  Every product and partial sum is exact
// in the tensor core's FP32 accumulation up to its rounding of the running sum, which is what the float64 reference is
// compared to; |l / 7| is at most a sixth of |h|, so what the two small accumulators round hardly reaches the result.
//
// Kernel: persistent, one block per SM over the 128 x 128 tiles of C.  One thread feeds the pipeline with TMA
// (cp.async.bulk.tensor.2d, 128-byte swizzle, each load for this CTA alone) and runs ahead into the next tile, one
// thread issues the MMAs, four warps write the scales of every K-step into tensor memory (tcgen05.st), four (NVFP4) or
// eight (IF4) warps read the accumulators back (tcgen05.ld) and write C.  Every mbarrier wait is bounded in time: when a
// wait runs out the block raises an error word, stops issuing, frees its tensor memory and returns.
//
// What bounds it: power.  Back to back, the GPU is at its power cap and lowers the clock (IF4, 8192 x 14336 x 4096: 1450 MHz), so what counts is
// energy and, below the cap, the cycles in which no MMA runs.  An MMA takes 64 cycles whatever else the SM's memories do (bulk
// copies at 50, shared loads at 120, tensor-memory loads at 280 bytes per cycle beside it change nothing, and neither do commits),
// the copy engine brings 110 bytes per cycle and SM, and the tensor core queues two MMAs: what used to take 93 cycles per MMA was the issuing thread,
// busy for 470 cycles between the MMAs of two steps.  Operands and split included, back to back: IF4 2048 x 4096 x 4096 72.2 -> 64.2
// us, 1000 x 14336 x 4096 133 -> 122 us, 8192 x 14336 x 4096 845 -> 787 us.  (Nine MMAs per K-block: 1440 us for the largest.)  NVFP4 26.8, 45.6 and
// 324 us one tile at a time; such products take their tiles in pairs (abs_pair.cuh).
#include "../../include/abs_b200.h"
#include "abs_tc.cuh"
#include "abs_rows.cuh"
#include "abs_skinny.cuh"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <mutex>
#include <type_traits>

namespace absq {

// A pipeline stage (one K-step) holds KBOXES boxes of each of the PLANES planes of A and of B; 192 KiB of stages are on their way or in use.
// IF4 (two planes, one box: K = 256, 64 KiB) has three stages.  Plain NVFP4 issues one MMA per K-block, so the hand-overs of a step weigh
// more: its steps are two boxes long where K allows (K = 512, 64 KiB, three stages), else one box (32 KiB, six stages).
// The scales.  IF4: boxes of 16 bytes x 128 rows as they lie, in a ring of their own (with the codes in their stage: 821 us instead of 790 for
// 8192 x 14336 x 4096).  The copy engine takes about a cycle per row of a box
// whatever its width, so beside the boxes of codes of an NVFP4 step, which has a quarter of the MMAs, there is no room for that: there the
// scales are tiled first (sf_tile_kernel) and come through registers.
template <int PLANES, int KBOXES> constexpr int kStageBytes = 2 * PLANES * KBOXES * kPlaneBytes;
template <int PLANES, int KBOXES> constexpr int kStages = PLANES * KBOXES == 2 ? 3 : 6;
constexpr int kSfBufs = 3, kScaleBoxBytes = kTileM * (kStageK / 16);
template <int PLANES> constexpr int kSfRingBytes = PLANES == 2 ? kSfBufs * 2 * kScaleBoxBytes : 0;
// Epilogue warps: IF4, whose accumulators fill the tensor memory, takes eight, two per quarter of the accumulator lanes,
// that have everything in registers before they store (the MMAs of the next tile wait only for that); NVFP4 has two sets
// of accumulators and streams each through four warps.  A thread stores the columns of its row 32 bytes at a time, whole sectors, straight from its
// registers (store_columns16).  Turned through shared memory, so that an instruction writes four rows of 128 bytes, the products took longer: IF4 100 x
// 4096 x 512 8.0 -> 7.3 us, 2048 x 4096 x 4096 57.3 -> 56.0, 4096 x 4096 x 512 24.4 -> 22.3, FP32 27.8 -> 25.0, at the power cap 8192 x 14336 x 4096 791 -> 779;
// NVFP4 300 x 4096 x 4096 11.4 -> 11.0, 1000 x 4096 x 1024 8.8 -> 8.2, FP32 9.3 -> 8.6.
template <int PLANES> constexpr int kEpiWarps = PLANES == 2 ? 8 : 4;
template <int PLANES> constexpr int kGemmThreads = 32 * (2 + kEpiWarps<PLANES> + 4);
template <int PLANES, int KBOXES> constexpr int kGemmSmemBytes =
    kStages<PLANES, KBOXES> * kStageBytes<PLANES, KBOXES> + kSfRingBytes<PLANES> + 1024 /* alignment slack */ + 512 /* barriers */;

// ----------------------------------------------------------------------------- operand split

// One operand of an IF4 product as the split kernel sees it.
struct SplitOperand {
    const uint4* codes;            // [rows, k / 2] bytes as abs_quantize wrote them
    const uint8_t* scales;         // [rows, k / 16] row-major
    uint4 *plane_h, *plane_l;
    int64_t pairs;                 // rows * k / 32: pairs of groups (16 bytes of codes)
};

// Writes the planes H and L of both operands of an IF4 product in one launch (an NVFP4 operand is read by the product kernel where it
// lies): 32 codes = two groups -> 16 bytes of each plane.  Also clears the error word.
__global__ void __launch_bounds__(256, 8) if4_split_kernel(const SplitOperand a, const SplitOperand b, int* __restrict__ error) {
    pdl_launch_dependents();
    pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (first == 0) { error[0] = 0; error[1] = 0; error[2] = 0; }     // error word, output maximum, ticket
    for (int64_t i = first; i < a.pairs + b.pairs; i += stride) {
        const SplitOperand& o = i < a.pairs ? a : b;
        const int64_t p = i < a.pairs ? i : i - a.pairs;
        const uint4 c = __ldg(o.codes + p);
        const uint32_t sb = __ldg(reinterpret_cast<const uint16_t*>(o.scales) + p);
        uint4 h = c, l = make_uint4(0u, 0u, 0u, 0u);
        if (sb & 0x80u) { split_int_word(c.x, h.x, l.x); split_int_word(c.y, h.y, l.y); }
        if (sb & 0x8000u) { split_int_word(c.z, h.z, l.z); split_int_word(c.w, h.w, l.w); }
        o.plane_h[p] = h;
        o.plane_l[p] = l;
    }
}

// The scales of both operands of an NVFP4 product in the 128x4-tile layout (16 bytes: the four K-blocks' bytes of rows r, r + 32, r + 64,
// r + 96 of a 128-row block): thread i of a warp reads 16 scale bytes of each of its four rows and writes 16 bytes of each of four
// consecutive tiles.  Also clears the error word.
struct TileOperand {
    const uint8_t* scales;         // [rows, k / 16] row-major
    uint8_t* tiled;
    int64_t rows;
    int64_t items;                 // ceil(rows / 128) * k / 256 * 32: one item = 4 rows x 16 scales
    uint32_t pitch, ksteps;        // k / 16, k / 256
};
__global__ void __launch_bounds__(256, 8) sf_tile_kernel(const TileOperand a, const TileOperand b, int* __restrict__ error) {
    pdl_launch_dependents();
    pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (first == 0) { error[0] = 0; error[1] = 0; error[2] = 0; }     // error word, output maximum, ticket
    for (int64_t i = first; i < a.items + b.items; i += stride) {
        const TileOperand& o = i < a.items ? a : b;
        const int64_t j = i < a.items ? i : i - a.items;
        const uint32_t lane = (uint32_t)(j & 31);
        const int64_t step = j >> 5;                                  // (row block, K-step)
        const uint32_t ksteps = o.ksteps;
        const int64_t rb = step / ksteps;
        const uint32_t kt = (uint32_t)(step - rb * ksteps);
        uint4 r[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t row = rb * 128 + q * 32 + lane;             // rows beyond the operand (last row block) get zero scales
            r[q] = row < o.rows ? __ldg(reinterpret_cast<const uint4*>(o.scales + row * o.pitch) + kt) : make_uint4(0u, 0u, 0u, 0u);
        }
        uint4* out = reinterpret_cast<uint4*>(o.tiled + ((size_t)rb * ksteps + kt) * 2048u) + lane;
        constexpr uint32_t kMag = 0x7F7F7F7Fu;
        out[0] = make_uint4(r[0].x & kMag, r[1].x & kMag, r[2].x & kMag, r[3].x & kMag);
        out[32] = make_uint4(r[0].y & kMag, r[1].y & kMag, r[2].y & kMag, r[3].y & kMag);
        out[64] = make_uint4(r[0].z & kMag, r[1].z & kMag, r[2].z & kMag, r[3].z & kMag);
        out[96] = make_uint4(r[0].w & kMag, r[1].w & kMag, r[2].w & kMag, r[3].w & kMag);
    }
}

// ----------------------------------------------------------------------------- the product kernel

// Tensor memory columns (512 allocated): the accumulators (IF4: three of 128 columns; NVFP4: two, used alternately),
// then the scale slots: 16 columns of A scales and 16 of B scales each (four per MMA of K = 64).
constexpr uint32_t kTmemCols = 512;

// Planes of A [M, K/2 bytes] and of B [N, K/2 bytes], boxes of 128 bytes x 128 rows: the codes (NVFP4), or H and L and, as abs_quantize wrote
// them, the scales [rows, K/16 bytes], boxes of 16 bytes x 128 rows (IF4).  sfa, sfb: the scales as sf_tile_kernel wrote them (NVFP4).
template <int PLANES> struct GemmMaps { CUtensorMap a[1], b[1]; const uint8_t *sfa, *sfb; };
template <> struct GemmMaps<2> { CUtensorMap a[2], b[2], sa, sb; };

// Tile t of the (tiles_m x tiles_n) grid of 128 x 128 tiles, walked in bands of eight tile rows, column by column
// inside a band, so that the blocks running at the same time share few rows of A and few of B (L2 reuse).
__device__ __forceinline__ void tile_of(int32_t t, int32_t tiles_m, int32_t tiles_n, int32_t& tm, int32_t& tn) {
    constexpr int32_t kBand = 8;
    const int32_t per_band = kBand * tiles_n, band = t / per_band, in_band = t - band * per_band;
    const int32_t first = band * kBand, rows = min(kBand, tiles_m - first);
    tn = in_band / rows;
    tm = first + (in_band - tn * rows);
}

// PLANES = 2: IF4 operands (four MMAs per K-block); PLANES = 1: plain NVFP4 (one).  error: device word set to a
// non-zero code when a wait ran out.
//
// Persistent: one block per SM walks the tiles blockIdx.x, blockIdx.x + gridDim.x, ...  Warp 0 (one thread) feeds the
// pipeline and runs ahead into the next tile while the current one is finished; warp 1 (one thread) issues MMAs; the next
// kEpiWarps warps are the epilogue (warp w reads the 32 accumulator lanes of tensor-memory quarter w % 4); the last four
// warps bring the scales of every K-step through registers to their quarter of tensor memory (tcgen05.st; every quarter holds the same four
// columns per MMA: rows r, r+32, r+64, r+96 of the tile); in IF4 a stage's full barrier counts them with the loads of its operands -- a
// tcgen05.cp from shared memory by the MMA thread would stand in the MMA queue for some 34 cycles per copy.  The accumulators pass between MMA and
// epilogue through acc_full / acc_empty barriers; NVFP4, with one accumulator of 128 columns, alternates between two of
// them so that a tile's epilogue overlaps the next tile's MMAs, IF4 (3 x 128 columns) has room for one set and overlaps
// only its stores and the next tile's loads.
// A block stays below the registers and the shared memory that would keep a block of the next call's split kernel from
// becoming resident beside it: without that overlap every call took 5 us longer.
// OUT_BF16: C is written as bf16 (round to nearest even of the same FP32 value), else as FP32.
template <int PLANES, bool OUT_BF16, int KBOXES = 1>
__global__ void __launch_bounds__(kGemmThreads<PLANES>, 1)
if4_gemm_kernel(const __grid_constant__ GemmMaps<PLANES> maps, const float* __restrict__ alpha_a, const float* __restrict__ alpha_b,
                void* __restrict__ c_out, int32_t tiles_m, int32_t tiles_n, int32_t k_iters, int32_t m_rows, int* __restrict__ error, int32_t stall_step,
                float* __restrict__ next_alpha, float next_denom) {
    constexpr int kStages = absq::kStages<PLANES, KBOXES>, kStageBytes = absq::kStageBytes<PLANES, KBOXES>;
    constexpr int kStepBlocks = KBOXES * (kStageK / kMmaK);          // MMA K-blocks (and scale tiles per operand) of one step
    constexpr int kAccBufs = PLANES == 1 ? 2 : 1;
    constexpr int kEpiWarps = absq::kEpiWarps<PLANES>;
    constexpr int kChunkSteps = PLANES == 2 ? kChunkK / kStageK : 1 << 30;    // NVFP4: the whole of K in one chain
    extern __shared__ uint8_t gemm_smem_raw[];
    const uint32_t raw = smem_u32(gemm_smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;                    // 128-byte swizzle wants 1024-byte aligned tiles
    // Scales in tensor memory: slots behind the accumulators (IF4: three, NVFP4: two), A scales, then B scales.
    constexpr uint32_t kSlotCols = 8u * kStepBlocks;                  // 4 columns per K-block and operand
    constexpr uint32_t kSfBase = PLANES == 1 ? 2 * kTileN : 3 * kTileN;
    // IF4: a slot per stage, NVFP4: as many as fit (four of a two-box step, eight of a one-box step)
    constexpr uint32_t kSfSlots = PLANES == 1 ? (kTmemCols - kSfBase) / kSlotCols : (uint32_t)kStages;
    static_assert(kSfBase + kSfSlots * kSlotCols <= kTmemCols && kSfSlots <= 8, "tensor memory, barriers");
    // barriers: full[], empty[] (stages), acc_full[2], acc_empty[2], drained, sf_full[], sf_empty[] (scale boxes, slots); then the tmem address word
    const uint32_t sf0 = base + kStages * kStageBytes, bars = sf0 + kSfRingBytes<PLANES>;
    uint32_t* tmem_word = reinterpret_cast<uint32_t*>(gemm_smem_raw + (bars - raw) + 320);
    const uint32_t full0 = bars, empty0 = bars + 64, acc_full0 = bars + 128, acc_empty0 = bars + 144, drained = bars + 160;
    const uint32_t sf_full0 = bars + 192, sf_empty0 = bars + 256;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t num_tiles = tiles_m * tiles_n, n_cols = tiles_n * kTileN;

    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full0 + 8 * s, PLANES == 2 ? 1 + 4 : 1);     // loads of the operands; IF4: and scale warps
            mbar_init(empty0 + 8 * s, 1);
        }
        // IF4: boxes of scales, filled by loads and emptied by the scale warps; NVFP4: slots, filled by these and emptied by the MMAs
        for (int i = 0; i < (PLANES == 2 ? kSfBufs : (int)kSfSlots); ++i) {
            mbar_init(sf_full0 + 8 * i, PLANES == 2 ? 1 : 4);
            mbar_init(sf_empty0 + 8 * i, PLANES == 2 ? 4 : 1);
        }
        for (int i = 0; i < kAccBufs; ++i) { mbar_init(acc_full0 + 8 * i, 1); mbar_init(acc_empty0 + 8 * i, kEpiWarps); }
        mbar_init(drained, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) { tmem_alloc(smem_u32(tmem_word), kTmemCols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, *tmem_word, 0);
    pdl_wait();

    if (warp == 0) {
        if (lane == 0) {
            // ---- producer: TMA loads of the operand planes
            uint32_t it = 0;
            bool ok = true;
            for (int32_t t = blockIdx.x; t < num_tiles && ok; t += gridDim.x) {
                int32_t tile_m, tile_n;
                tile_of(t, tiles_m, tiles_n, tile_m, tile_n);
                for (int32_t kt = 0; kt < k_iters; ++kt, ++it) {
                    const bool stalled = (int32_t)it == stall_step;      // self-test only: the bytes announced never arrive
                    if constexpr (PLANES == 2) {
                        const uint32_t b = it % kSfBufs, at = sf0 + b * 2 * kScaleBoxBytes, bar = sf_full0 + 8 * b;
                        if (!mbar_wait(sf_empty0 + 8 * b, ((it / kSfBufs) & 1u) ^ 1u)) { atomicExch(error, 7); ok = false; break; }
                        mbar_expect_tx(bar, 2 * kScaleBoxBytes);
                        if (!stalled) {
                            tma_load_2d(at, &maps.sa, kt * (kStageK / 16), tile_m * kTileM, bar);
                            tma_load_2d(at + kScaleBoxBytes, &maps.sb, kt * (kStageK / 16), tile_n * kTileN, bar);
                        }
                    }
                    const uint32_t s = it % kStages;
                    if (!mbar_wait(empty0 + 8 * s, ((it / kStages) & 1u) ^ 1u)) { atomicExch(error, 1); ok = false; break; }
                    const uint32_t st = base + s * kStageBytes, bar = full0 + 8 * s;
                    mbar_expect_tx(bar, kStageBytes);
                    if (stalled) continue;
#pragma unroll
                    for (int p = 0; p < PLANES; ++p)
#pragma unroll
                        for (int box = 0; box < KBOXES; ++box) {
                            const int32_t x = (kt * KBOXES + box) * (kStageK / 2);
                            tma_load_2d(st + (p * KBOXES + box) * kPlaneBytes, &maps.a[p], x, tile_m * kTileM, bar);
                            tma_load_2d(st + ((PLANES + p) * KBOXES + box) * kPlaneBytes, &maps.b[p], x, tile_n * kTileN, bar);
                        }
                }
            }
        }
    } else if (warp == 1) {
        if (PLANES == 2 && lane == 0) {
            // ---- MMAs.  The tensor core's queue holds about two MMAs of 64 cycles, so what this thread does between two of them must
            // take less than that: descriptors by one addition, stages and parities kept and not computed, and the wait for the next step's
            // operands in the middle of this step's MMAs.  (Warp-wide loop with votes, remainders, and the wait after the step's MMAs: 470 cycles
            // a step without an MMA running.)
            const uint64_t desc0 = operand_desc(base);
            uint32_t s = 0, parity = 0, j = 0;          // stage and its parity; chunks so far
            bool ok = mbar_wait(full0, 0);
            for (int32_t t = blockIdx.x, k0 = 0; t < num_tiles && ok; ++j) {
                const uint32_t buf = j % kAccBufs, acc = tmem + buf * kTileN;
                if (!mbar_wait(acc_empty0 + 8 * buf, ((j / kAccBufs) & 1u) ^ 1u)) { atomicExch(error, 4); break; }
                tc_fence_after();
                const int32_t k_end = min(k_iters - k0, kChunkSteps);
                const bool last_chunk = k0 + k_end == k_iters && t + (int32_t)gridDim.x >= num_tiles;
                for (int32_t kt = 0; kt < k_end; ++kt) {
                    const uint32_t s1 = s + 1 == kStages ? 0u : s + 1, parity1 = s1 ? parity : parity ^ 1u;
                    const uint64_t st = desc0 + (uint64_t)s * (kStageBytes >> 4);
                    const uint32_t tsfa = tmem + kSfBase + s * kSlotCols, tsfb = tsfa + kSlotCols / 2;
                    const bool first = kt == 0, go = !first || k0 != 0;           // H H: anew in every chunk
                    // 32 bytes per K-block inside a box's 128-byte rows
                    auto mmas = [&](int kb) __attribute__((always_inline)) {
                        constexpr uint64_t L = kPlaneBytes >> 4;
                        const uint64_t a = st + ((kb * (kMmaK / 2)) >> 4), b = a + 2 * L;
                        const uint32_t fa = tsfa + 4 * kb, fb = tsfb + 4 * kb;
                        tc_mma_nvf4<kFill>(acc, a, b, kInstrDesc, kb > 0 || !first, fa, fb);                     // H H
                        tc_mma_nvf4<kLastUse>(acc + kTileN, a, b + L, kInstrDesc, kb > 0 || go, fa, fb);         // H L
                        tc_mma_nvf4<kFill>(acc + kTileN, a + L, b, kInstrDesc, true, fa, fb);                    // L H
                        tc_mma_nvf4<kLastUse>(acc + 2 * kTileN, a + L, b + L, kInstrDesc, kb > 0 || go, fa, fb); // L L
                    };
                    constexpr int kBefore = kStepBlocks - 1;
#pragma unroll
                    for (int kb = 0; kb < kBefore; ++kb) mmas(kb);
                    // The next step's stage was handed back kStages - 1 commits ago, so this waits for loads and scales alone.
                    if (!(last_chunk && kt == k_end - 1)) ok = mbar_wait(full0 + 8 * s1, parity1);
                    if (!ok) break;                     // nothing more is issued, and the chunk is not handed over
                    tc_fence_after();
#pragma unroll
                    for (int kb = kBefore; kb < kStepBlocks; ++kb) mmas(kb);
                    tc_commit(empty0 + 8 * s);          // the stage's shared memory and scales are free once these MMAs have run
                    s = s1;
                    parity = parity1;
                }
                if (ok) tc_commit(acc_full0 + 8 * buf); // and the chunk's accumulators are complete
                k0 += k_end;
                if (k0 == k_iters) { k0 = 0; t += gridDim.x; }
            }
            if (!ok) atomicExch(error, 2);
        }
        if (PLANES == 1 && lane == 0) {
            // ---- MMAs, NVFP4.  With the loop above and a second group of scale warps, which it needs, products back to back take 4 % less (45.6 ->
            // 43.5 us), but a pass with its quantizers more (1000 x 14336 x 4096 chained 55.9 -> 58.0 us, a layer's backward pass 133.4 -> 135.1):
            // the next kernel's blocks find less room beside the larger block.
            uint32_t it = 0, j = 0;                     // K-steps and chunks so far
            bool ok = true;
            for (int32_t t = blockIdx.x, k0 = 0; t < num_tiles && ok; ++j) {
                const uint32_t buf = j % kAccBufs, acc = tmem + buf * kTileN;
                if (!mbar_wait(acc_empty0 + 8 * buf, ((j / kAccBufs) & 1u) ^ 1u)) { atomicExch(error, 4); ok = false; break; }
                tc_fence_after();
                const int32_t k_end = min(k_iters - k0, kChunkSteps);
                for (int32_t kt = 0; kt < k_end; ++kt, ++it) {
                    const uint32_t s = it % kStages;
                    const uint32_t slot = it % kSfSlots;
                    if (!mbar_wait(full0 + 8 * s, (it / kStages) & 1u)) { atomicExch(error, 2); ok = false; break; }
                    if (!mbar_wait(sf_full0 + 8 * slot, (it / kSfSlots) & 1u)) { atomicExch(error, 5); ok = false; break; }
                    tc_fence_after();
                    const uint32_t st = base + s * kStageBytes;
                    const uint32_t tsfa = tmem + kSfBase + slot * kSlotCols, tsfb = tsfa + kSlotCols / 2;
                    // K-block kb of a step lies in box kb / 4 of its plane, 32 bytes per K-block inside the box's 128-byte rows
                    auto desc_a = [&](int kb) { return operand_desc(st + (kb >> 2) * kPlaneBytes + (kb & 3) * (kMmaK / 2)); };
                    auto desc_b = [&](int kb) { return operand_desc(st + (KBOXES + (kb >> 2)) * kPlaneBytes + (kb & 3) * (kMmaK / 2)); };
#pragma unroll
                    for (int kb = 0; kb < kStepBlocks; ++kb)
                        tc_mma_nvf4(acc, desc_a(kb), desc_b(kb), kInstrDesc, !(kt == 0 && kb == 0), tsfa + 4 * kb, tsfb + 4 * kb);
                    tc_commit(empty0 + 8 * s);          // the stage's shared memory is free once these MMAs have run
                    tc_commit(sf_empty0 + 8 * slot);    // and so is the slot of scales
                }
                if (ok) tc_commit(acc_full0 + 8 * buf); // and the chunk's accumulators are complete
                k0 += k_end;
                if (k0 == k_iters) { k0 = 0; t += gridDim.x; }
            }
        }
        if (lane == 0) {
            // All MMAs are over before the block frees its tensor memory, also where the epilogue has given up and waits for none of them.
            tc_commit(drained);
            if (!mbar_wait(drained, 0)) atomicExch(error, 8);
        }
    } else if (warp >= 2 + kEpiWarps) {
        // ---- scales: this warp's copy of every K-step's scales, through registers into tensor memory
        const uint32_t lane_base = tmem + kSfBase + ((uint32_t)((warp & 3) * 32) << 16);
        if constexpr (PLANES == 2) {
            const uint32_t steps = (uint32_t)((num_tiles - (int32_t)blockIdx.x + (int32_t)gridDim.x - 1) / (int32_t)gridDim.x) * (uint32_t)k_iters;
            for (uint32_t it = 0; it < steps; ++it) {
                const uint32_t s = it % kStages, bx = it % kSfBufs;
                const bool ok = mbar_wait_warp(sf_full0 + 8 * bx, (it / kSfBufs) & 1u) && mbar_wait_warp(empty0 + 8 * s, ((it / kStages) & 1u) ^ 1u);
                if (!ok) { if (lane == 0) atomicExch(error, 6); break; }
                // 16 scale bytes (four K-blocks) of each of the rows r, r + 32, r + 64, r + 96 of either operand, flag bits stripped
                const uint4* at = reinterpret_cast<const uint4*>(gemm_smem_raw + (sf0 - raw) + bx * 2 * kScaleBoxBytes) + lane;
                tc_fence_after();
#pragma unroll
                for (int op = 0; op < 2; ++op) {
                    const uint4 r0 = at[op * 128], r1 = at[op * 128 + 32], r2 = at[op * 128 + 64], r3 = at[op * 128 + 96];
                    tmem_store16(lane_base + s * kSlotCols + op * (kSlotCols / 2), mask_scales(r0.x, r1.x, r2.x, r3.x), mask_scales(r0.y, r1.y, r2.y, r3.y),
                                 mask_scales(r0.z, r1.z, r2.z, r3.z), mask_scales(r0.w, r1.w, r2.w, r3.w));
                }
                tmem_store_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) { mbar_arrive(full0 + 8 * s); mbar_arrive(sf_empty0 + 8 * bx); }
            }
        } else {
            // The loads of step it + 1 are in flight while step it waits for its slot and is written.
            const int32_t ktiles = k_iters * kStepBlocks;
            int32_t t = blockIdx.x, kt = 0;                                   // the step whose tiles are loaded next
            const uint4 *pa = nullptr, *pb = nullptr;
            auto load_next = [&](uint4 (&a)[kStepBlocks], uint4 (&b)[kStepBlocks]) {   // false when there is no further step
                if (t >= num_tiles) return false;
                if (kt == 0) {
                    int32_t tile_m, tile_n;
                    tile_of(t, tiles_m, tiles_n, tile_m, tile_n);
                    pa = reinterpret_cast<const uint4*>(maps.sfa + (size_t)tile_m * ktiles * 512) + lane;
                    pb = reinterpret_cast<const uint4*>(maps.sfb + (size_t)tile_n * ktiles * 512) + lane;
                }
#pragma unroll
                for (int kb = 0; kb < kStepBlocks; ++kb) {                     // tile kb of the step: 16 bytes per lane, tiles 512 bytes apart
                    a[kb] = __ldg(pa + (kt * kStepBlocks + kb) * 32);
                    b[kb] = __ldg(pb + (kt * kStepBlocks + kb) * 32);
                }
                if (++kt == k_iters) { kt = 0; t += gridDim.x; }
                return true;
            };
            // One step of lookahead in registers where a step is one box long; with two-box steps the four scale slots
            // already let these warps run three steps ahead of the MMAs.
            constexpr bool kLookahead = KBOXES == 1;
            uint4 a[kStepBlocks], b[kStepBlocks], an[kLookahead ? kStepBlocks : 1], bn[kLookahead ? kStepBlocks : 1];
            bool more = load_next(a, b);
            for (uint32_t it = 0; more; ++it) {
                if constexpr (kLookahead) more = load_next(an, bn);
                const uint32_t slot = it % kSfSlots;
                bool have = mbar_wait(sf_empty0 + 8 * slot, ((it / kSfSlots) & 1u) ^ 1u);
                if (!have && lane == 0) atomicExch(error, 6);
                have = __all_sync(0xFFFFFFFFu, have);
                if (!have) break;
                tc_fence_after();
#pragma unroll
                for (int g = 0; g < KBOXES; ++g) {
                    tmem_store16(lane_base + slot * kSlotCols + 16u * g, a[4 * g], a[4 * g + 1], a[4 * g + 2], a[4 * g + 3]);
                    tmem_store16(lane_base + slot * kSlotCols + kSlotCols / 2 + 16u * g, b[4 * g], b[4 * g + 1], b[4 * g + 2], b[4 * g + 3]);
                }
                tmem_store_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(sf_full0 + 8 * slot);
                if constexpr (kLookahead) {
#pragma unroll
                    for (int kb = 0; kb < kStepBlocks; ++kb) { a[kb] = an[kb]; b[kb] = bn[kb]; }
                } else {
                    more = load_next(a, b);
                }
            }
        }
    } else {
        // ---- epilogue
        const int quarter = warp & 3;
        const float scale = __fmul_rn(__ldg(alpha_a), __ldg(alpha_b));
        uint32_t j = 0;
        uint32_t out_max = 0u;                  // bf16 output with next_alpha: largest |C| bit patterns this thread has written (see store_columns16)
        const bool out_aligned32 = (reinterpret_cast<uintptr_t>(c_out) & 31u) == 0;
        uint4 held = make_uint4(0u, 0u, 0u, 0u);   // see store_columns16
        bool all_tiles = true;
        if constexpr (PLANES == 2) {
            // Two warps per quarter of tensor memory; a warp owns the accumulator lanes (rows of the tile) 32 (w % 4) ..
            // 32 (w % 4) + 31 of one half (64) of the columns.  It takes its share into registers, hands the accumulators
            // back, and only then stores.
            constexpr int kCols = kTileN / 2;
            const int col0 = ((warp - 2) >> 2) * kCols;
            const float c1 = __uint_as_float(0x3E124925u), c2 = __uint_as_float(0x3CA72F05u);      // fp32(1/7), fp32(1/49)
            for (int32_t t = blockIdx.x; t < num_tiles && all_tiles; t += gridDim.x) {
                int32_t tile_m, tile_n;
                tile_of(t, tiles_m, tiles_n, tile_m, tile_n);
                const bool own_row_valid = tile_m * kTileM + quarter * 32 + lane < m_rows;   // the row whose values this thread holds
                const size_t first = (size_t)(tile_m * kTileM + quarter * 32 + lane) * (size_t)n_cols + (size_t)tile_n * kTileN + col0;
                float v[kCols];
                for (int32_t k0 = 0; k0 < k_iters; k0 += kChunkSteps, ++j) {
                    const uint32_t buf = j % kAccBufs;
                    bool have = mbar_wait(acc_full0 + 8 * buf, (j / kAccBufs) & 1u);
                    if (!have && lane == 0) atomicExch(error, 3);
                    have = __all_sync(0xFFFFFFFFu, have);
                    if (!have) { all_tiles = false; break; }
                    tc_fence_after();
                    const uint32_t lane_base = tmem + buf * kTileN + col0 + ((uint32_t)(quarter * 32) << 16);
                    // H H of a chunk is added to that of the chunks before it; the other two accumulators run on to the last (see kChunkK)
#pragma unroll
                    for (int chunk = 0; chunk < kCols / 16; ++chunk) {
                        uint32_t r0[16];
                        tmem_load16(lane_base + chunk * 16, r0);
                        tmem_load_wait();
#pragma unroll
                        for (int jj = 0; jj < 16; ++jj)
                            v[chunk * 16 + jj] = k0 == 0 ? __uint_as_float(r0[jj]) : __fadd_rn(v[chunk * 16 + jj], __uint_as_float(r0[jj]));
                    }
                    if (k_iters - k0 <= kChunkSteps) {
#pragma unroll
                        for (int chunk = 0; chunk < kCols / 16; ++chunk) {
                            uint32_t r1[16], r2[16];
                            tmem_load16(lane_base + kTileN + chunk * 16, r1);
                            tmem_load16(lane_base + 2 * kTileN + chunk * 16, r2);
                            tmem_load_wait();
#pragma unroll
                            for (int jj = 0; jj < 16; ++jj)
                                v[chunk * 16 + jj] = __fadd_rn(v[chunk * 16 + jj], __fmaf_rn(c2, __uint_as_float(r2[jj]), __fmul_rn(c1, __uint_as_float(r1[jj]))));
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acc_empty0 + 8 * buf);    // the MMAs of the next chunk or tile may start
                }
                if (!all_tiles) break;
                if (own_row_valid) {
#pragma unroll
                    for (int q = 0; q < kCols / 16; ++q) {
                        if (out_aligned32) store_columns16<OUT_BF16, true>(c_out, first + 16 * q, v + 16 * q, scale, false, false, held, next_alpha != nullptr, out_max);
                        else store_columns16<OUT_BF16, false>(c_out, first + 16 * q, v + 16 * q, scale, q == 0, q == kCols / 16 - 1, held, next_alpha != nullptr, out_max);
                    }
                }
            }
        } else {
            // A warp owns the accumulator lanes (rows of the tile) 32 (w % 4) .. 32 (w % 4) + 31.
            for (int32_t t = blockIdx.x; t < num_tiles; t += gridDim.x, ++j) {
                int32_t tile_m, tile_n;
                tile_of(t, tiles_m, tiles_n, tile_m, tile_n);
                const uint32_t buf = j % kAccBufs;
                bool have = mbar_wait(acc_full0 + 8 * buf, (j / kAccBufs) & 1u);
                if (!have && lane == 0) atomicExch(error, 3);
                have = __all_sync(0xFFFFFFFFu, have);
                if (!have) { all_tiles = false; break; }
                tc_fence_after();
                const bool own_row_valid = tile_m * kTileM + quarter * 32 + lane < m_rows;   // the row whose values this thread holds
                const size_t first = (size_t)(tile_m * kTileM + quarter * 32 + lane) * (size_t)n_cols + (size_t)tile_n * kTileN;
                const uint32_t lane_base = tmem + buf * kTileN + ((uint32_t)(quarter * 32) << 16);
                for (int chunk = 0; chunk < kTileN / 32; ++chunk) {
                    uint32_t r0[32];
                    tmem_load32(lane_base + chunk * 32, r0);
                    tmem_load_wait();
                    if (chunk == kTileN / 32 - 1) {         // everything is in registers: the MMAs of the next tile may start
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(acc_empty0 + 8 * buf);
                    }
                    float v[32];
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj) v[jj] = __uint_as_float(r0[jj]);
                    const auto store = [&](auto whole) __attribute__((always_inline)) {
#pragma unroll
                        for (int q = 0; q < 2; ++q)
                            store_columns16<OUT_BF16, decltype(whole)::value>(c_out, first + chunk * 32 + 16 * q, v + 16 * q, scale, chunk + q == 0,
                                                                              chunk == kTileN / 32 - 1 && q == 1, held, next_alpha != nullptr, out_max);
                    };
                    if (own_row_valid) {
                        if (out_aligned32) store(std::true_type{});
                        else store(std::false_type{});
                    }
                }
            }
        }
        // The global maximum of |C| as written (bf16), for the next quantizer's tensor scale (Eq. 1): every epilogue
        // warp publishes its maximum with an atomic and takes a ticket; the last of all warps converts and writes alpha.
        if (OUT_BF16 && next_alpha != nullptr && all_tiles) {
            const uint32_t wmax = __reduce_max_sync(0xFFFFFFFFu, max(out_max & 0xFFFFu, out_max >> 16));
            if (lane == 0) {
                atomicMax(reinterpret_cast<unsigned int*>(error) + 1, wmax);
                __threadfence();
                const int ticket = atomicAdd(error + 2, 1);
                if (ticket == (int)gridDim.x * kEpiWarps - 1) {
                    const float A = __uint_as_float(atomicMax(reinterpret_cast<unsigned int*>(error) + 1, 0u) << 16);
                    *next_alpha = (A == 0.0f) ? 1.0f : __fdiv_rn(A, next_denom);
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, kTmemCols);
}

}  // namespace absq

#include "abs_pair.cuh"

// ----------------------------------------------------------------------------- host side

namespace {

using namespace absq;

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled through the runtime's driver entry point (the library does not link libcuda).
EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, []() {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// Tensor map of one plane: bytes [rows, row_bytes], box 128 bytes x 128 rows, 128-byte swizzle.  The map covers
// this GPU's own workspace only.
bool plane_map(CUtensorMap* map, void* base, uint64_t rows, uint64_t row_bytes) {
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    const cuuint64_t dims[2] = {row_bytes, rows};
    const cuuint64_t strides[1] = {row_bytes};
    const cuuint32_t box[2] = {128, 128}, elem[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, base, dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tensor map of row-major scales: bytes [rows, row_bytes], box 16 bytes x 128 rows, no swizzle.
bool scale_map(CUtensorMap* map, void* base, uint64_t rows, uint64_t row_bytes) {
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    const cuuint64_t dims[2] = {row_bytes, rows};
    const cuuint64_t strides[1] = {row_bytes};
    const cuuint32_t box[2] = {16, 128}, elem[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, base, dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t round1k(size_t n) { return (n + 1023) & ~(size_t)1023; }

// Launch with programmatic stream serialization: the kernel may become resident while its predecessor in the stream
// drains; every kernel launched so calls pdl_wait() before it reads or writes global memory (requests into the L2 consume nothing and may come before).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
constexpr int kMaxSms = 160;               // workspaces are sized for up to this many SMs
// Workspace of the tiled kernel behind the header: planes H, L of A, then of B (IF4); tiled scales of A, then of B (NVFP4).
struct GemmLayout {
    size_t plane_a, plane_b;                   // size of one plane (IF4)
    size_t off_a, off_b, total;
};
GemmLayout gemm_layout(abs_fmt_t fmt, int64_t m, int64_t n, int64_t k) {
    GemmLayout L;
    L.plane_a = round1k((size_t)m * k / 2);
    L.plane_b = round1k((size_t)n * k / 2);
    const size_t sf_a = round1k((size_t)((m + kTileM - 1) / kTileM * kTileM) * k / 16), sf_b = round1k((size_t)n * k / 16);
    L.off_a = 1024;
    L.off_b = L.off_a + (fmt == ABS_FMT_IF4 ? 2 * L.plane_a : sf_a);
    L.total = L.off_b + (fmt == ABS_FMT_IF4 ? 2 * L.plane_b : sf_b);
    return L;
}

// Plan and workspace of the product with few rows of A (see abs_skinny.cuh): tickets, partial sums.
struct SkinnyPlan {
    int32_t units, grid;
    size_t off_partials, total;
};
// The rule: IF4 with up to 32 rows of A, except, with more than 8 rows, where the whole of B is fewer than 64 steps, which the blocks of this file's
// kernel take in one go (1024 x 1024, 16 rows: 8.9 us there, 9.5 here).  With up to 8 rows such a B comes here where K is too long for
// abs_rows.cuh: 8 x 128 x 14336 14.1 us, 41 us there.  With 33 to 64 rows (64 columns for the MMA's N side, two stages) it lost at every size
// below 8192 x 8192.  NVFP4 has no planes to save and measured slower at all sizes.
bool skinny_plan(abs_fmt_t fmt, int64_t m, int64_t n, int64_t k, int sm_count, SkinnyPlan& P) {
    const int64_t units = n / kTileM * (k / kStageK);
    if (fmt != ABS_FMT_IF4 || m > kSkinnyMaxRows || (m > 8 && units < 64) || units > 0x7FFFFFFF) return false;
    P.units = (int32_t)units;
    P.grid = P.units < sm_count ? P.units : sm_count;
    P.off_partials = 1024 + round1k((size_t)(n / kTileM) * sizeof(int));
    P.total = P.off_partials + (size_t)P.grid * 2 * kSkinnyTok * kTileM * sizeof(double);
    return true;
}

// The product with very few rows of A (see abs_rows.cuh).
int rows_instance(int64_t m) { return m <= 1 ? 1 : m <= 2 ? 2 : m <= 4 ? 4 : 8; }
// The blocks of it that fit on an SM.
int rows_blocks_fit(int64_t m, int64_t k) {
    const int64_t fit = kRowsMaxSmem / (int64_t)rows_smem_bytes(rows_instance(m), k);
    return (int)(fit < rows_blocks(rows_instance(m)) ? fit : rows_blocks(rows_instance(m)));
}
// The rule.  What the kernel does is turns (two rows of B) per warp times chunks of K; a warp that has one turn walks the whole of K by itself, and
// a block lays out all tokens, so chunks are dear and rows of B are cheap until all warps have some.  The kernels beside it split K over
// the SMs (IF4, abs_skinny.cuh) or have a chain that grows with K, twice as steep where K is no multiple of 512 (NVFP4, abs_gemm.cu).  Measured at 14477
// points, n = 128 .. 32768, K = 256 .. 16384, 1, 2, 4 and 8 rows, chained and not; the lines are where this kernel is no longer the faster one
// (of the 9818 points that it takes with K >= 1024 and n <= 14336 it is more than 3 % slower at 50, 13 % at the worst; over all points there the choice
// costs 0.3 % against the faster of both).
//   IF4, warps with one turn: 1 row 4096 x 14336 15.8 / 18.6, 128 x 32768 21.1 / 18.5; 2 rows 4096 x 10240 13.6 / 15.3, 1024 x 14336 14.0 / 12.6; 4 rows
//   7168 x 5120 13.8 / 14.7, 1024 x 14336 17.3 / 13.1; 8 rows 4096 x 4096 10.4 / 12.5, 4096 x 8192 24.5 / 14.9, 512 x 14336 20.0 / 13.7.
//   IF4, more turns: 1 row 14336 x 8192 27.1 / 27.7, 14336 x 14336 46.5 / 43.3; 2 rows 14336 x 4096 14.8 / 17.5, 14336 x 8192 29.8 / 27.8; 4 rows 14336 x
//   1280 10.3 / 11.0, 9472 x 4096 14.3 / 13.3; 8 rows 7168 x 1280 9.1 / 9.8, 7168 x 2304 12.6 / 11.3.
//   NVFP4: 1 row 14336 x 14336 43.6 / 53.2; 4 rows 4096 x 8192 13.3 / 15.9, 12800 x 1280 9.6 / 8.7; 8 rows 4096 x 4096 10.1 / 10.9, 7168 x 2304 12.2 / 10.4,
//   2048 x 7424 13.5 / 18.7, 3072 x 7168 14.6 / 12.8.
// (At K = 256 the other kernels take 5 us whatever n; a quarter of the turns less.)  The rule does not ask for the type of the output or for a next
// tensor scale, though the latter costs this kernel a launch and an atomic per warp: the bf16 outputs are the FP32 ones rounded.
bool rows_rule(abs_fmt_t fmt, int64_t m, int64_t n, int64_t k, int sm_count) {
    if (m > kRowsMax || n * k > 224000000 / rows_instance(m) || rows_smem_bytes(rows_instance(m), k) > (size_t)kRowsMaxSmem) return false;
    const bool has_int = fmt == ABS_FMT_IF4;
    const int i = m <= 1 ? 0 : m <= 2 ? 1 : m <= 4 ? 2 : 3;                                        // instance
    const int64_t chunks = (k + kRowsChunk - 1) / kRowsChunk, turns = n / kRowsPerTurn;
    const int64_t warps = (int64_t)sm_count * rows_blocks_fit(m, k) * kRowsWarps;
    if (k == kStageK) return 4 * turns < 3 * warps;
    if (turns * (has_int ? 128 : 500) > warps * k) return false;
    if (has_int) {
        static const int half[4] = {14, 10, 8, 6}, one[4] = {14, 10, 6, 5}, more[4] = {110, 77, 45, 35};
        if (turns < warps) return chunks <= (2 * turns < warps ? half : one)[i];
        return 10 * turns * chunks <= more[i] * warps;
    }
    if (m <= 2) return true;
    if (64 * turns > 65 * warps)
        return (m <= 4 && chunks <= 10 && 2 * turns < 3 * warps) || 10 * kRowsChunk * turns * chunks * chunks <= (m <= 4 ? 43 : 30) * warps * k;
    return m <= 4 || k % (2 * kStageK) != 0 || n * chunks <= (int64_t)kTileN * sm_count;
}
// NVFP4: which products take their tiles in pairs (abs_pair.cuh) and not one by one: those that need no more rounds so (an odd number of tile columns leaves
// pairs of one tile, and the last round is one of pairs or of single tiles), with more than one round and a long K, where the feed counts, or with three
// rounds or more, where the overlap of the ends does too (FP32, whose stores weigh more, from K = 1024 on).  One by one / in pairs, us, bf16 and FP32:
// 600 x 4096 x 1024 (160 tiles) 8.0 / 8.6, 8.5 / 9.1; 1000 x 4096 x 2048 (256) 10.7 / 10.8, 11.1 / 11.5; 1000 x 4096 x 3072 12.9 / 12.6, 13.9 / 13.4; 300 x 14336 x
// 1024 (336) 10.0 / 10.1, 10.6 / 11.5; 2048 x 4096 x 512 (512) 9.7 / 9.5, 11.3 / 11.5; 2048 x 4096 x 2048 15.9 / 15.3, 17.9 / 17.3; 1000 x 14336 x 256 (896)
// 12.5 / 11.4, 15.3 / 15.9; 1000 x 14336 x 1024 16.6 / 15.6, 20.1 / 19.5; 3000 x 4736 x 2048 (888; six rounds or seven) 21.1 / 22.6, 25.0 / 27.7; back to back for
// longer, at the power cap, 8192 x 14336 x 4096 321 / 274, 388 / 326.
bool pair_rule(bool out_bf16, int64_t tiles_m, int64_t tiles_n, int64_t k, int sm_count) {
    const int64_t tiles = tiles_m * tiles_n, pairs = tiles_m * ((tiles_n + 1) / 2), rest = pairs % sm_count;
    if (tiles <= sm_count || (k < 3072 && (tiles < 3 * (int64_t)sm_count || !(out_bf16 || k >= 1024)))) return false;
    return pairs / sm_count * 2 + (rest == 0 ? 0 : 2 * rest <= sm_count ? 1 : 2) <= (tiles + sm_count - 1) / sm_count;
}
typedef void (*RowsKernel)(RowsArgs);
template <int M> RowsKernel rows_kernel_for(bool has_int, bool out_bf16) {
    return has_int ? (out_bf16 ? rows_kernel<M, true, true> : rows_kernel<M, true, false>)
                   : (out_bf16 ? rows_kernel<M, false, true> : rows_kernel<M, false, false>);
}
RowsKernel rows_kernel_of(int64_t m, bool has_int, bool out_bf16) {
    switch (rows_instance(m)) {
        case 1: return rows_kernel_for<1>(has_int, out_bf16);
        case 2: return rows_kernel_for<2>(has_int, out_bf16);
        case 4: return rows_kernel_for<4>(has_int, out_bf16);
        default: return rows_kernel_for<8>(has_int, out_bf16);
    }
}

bool gemm_shape_ok(abs_fmt_t fmt, int64_t m, int64_t n, int64_t k) {
    return (fmt == ABS_FMT_IF4 || fmt == ABS_FMT_NVFP4) && m > 0 && n > 0 && k > 0 && n % kTileN == 0 &&
           k % kStageK == 0 && m < ((int64_t)1 << 30) && n < ((int64_t)1 << 30) && k < ((int64_t)1 << 30);
}

}  // namespace

extern "C" {

size_t abs_matmul_workspace_bytes(abs_fmt_t fmt, int64_t m, int64_t n, int64_t k) {
    if (!gemm_shape_ok(fmt, m, n, k)) return 0;
    // For the largest grid: the size must not depend on the device that happens to be current (which kernel runs does not).  A
    // workspace for many rows also serves fewer: programs take one for their largest m.
    SkinnyPlan P;
    if (skinny_plan(fmt, m, n, k, kMaxSms, P)) return P.total;
    const size_t total = gemm_layout(fmt, m, n, k).total;
    return skinny_plan(fmt, 1, n, k, kMaxSms, P) && P.total > total ? P.total : total;
}

// The product with few rows of A.  Arguments are already validated.
static abs_status_t skinny_matmul(const SkinnyPlan& P, const void* a_codes, const void* a_scales, const float* a_alpha,
                                  const void* b_codes, const void* b_scales, const float* b_alpha, int64_t m, int64_t n, int64_t k,
                                  void* out, uint8_t* ws, cudaStream_t s, int32_t stall_step, bool out_bf16, float* next_alpha, float next_denom) {
    SkinnyArgs p;
    if (!plane_map(&p.w_codes, const_cast<void*>(b_codes), (uint64_t)n, (uint64_t)k / 2) ||
        !scale_map(&p.w_scales, const_cast<void*>(b_scales), (uint64_t)n, (uint64_t)k / 16))
        return ABS_ERR_CUDA;
    p.x_codes = (const uint8_t*)a_codes; p.x_scales = (const uint8_t*)a_scales;
    p.alpha_a = a_alpha; p.alpha_b = b_alpha;
    p.out = out;
    p.partials = (double*)(ws + P.off_partials);
    p.tickets = (int*)(ws + 1024); p.error = (int*)ws;
    p.m = (int32_t)m; p.n = (int32_t)n; p.k = (int32_t)k; p.units = P.units; p.stall_step = stall_step;
    p.next_alpha = next_alpha; p.next_denom = next_denom;
    if (launch_pdl(skinny_clear_kernel, dim3(1), 256, 0, s, (int*)ws, p.tickets, (int32_t)(n / kTileM)) != cudaSuccess) return ABS_ERR_CUDA;
    const cudaError_t e = launch_pdl(out_bf16 ? skinny_kernel<true> : skinny_kernel<false>, dim3((unsigned)P.grid), kSkinnyThreads,
                                     kSkinnySmemBytes, s, p);
    if (e != cudaSuccess) return ABS_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? ABS_OK : ABS_ERR_CUDA;
}

// The product with very few rows of A.  Arguments are already validated.
static abs_status_t rows_matmul(bool has_int, const void* a_codes, const void* a_scales, const float* a_alpha, const void* b_codes,
                                const void* b_scales, const float* b_alpha, int64_t m, int64_t n, int64_t k, void* out, uint8_t* ws,
                                cudaStream_t s, int sm_count, bool out_bf16, float* next_alpha, float next_denom) {
    RowsArgs p;
    p.w_codes = (const uint8_t*)b_codes; p.w_scales = (const uint8_t*)b_scales;
    p.x_codes = (const uint8_t*)a_codes; p.x_scales = (const uint8_t*)a_scales;
    p.alpha_a = a_alpha; p.alpha_b = b_alpha;
    p.out = out; p.error = (int*)ws;
    p.m = (int32_t)m; p.n = (int32_t)n; p.k = (int32_t)k;
    p.next_alpha = next_alpha; p.next_denom = next_denom;
    // the maximum and its ticket start at zero; without them the kernel clears the error word itself
    if (next_alpha && launch_pdl(skinny_clear_kernel, dim3(1), 32, 0, s, (int*)ws, (int*)ws, 0) != cudaSuccess) return ABS_ERR_CUDA;
    const size_t smem = rows_smem_bytes(rows_instance(m), k);
    const int64_t turns = n / kRowsPerTurn, blocks = (int64_t)sm_count * rows_blocks_fit(m, k);
    if (launch_pdl(rows_kernel_of(m, has_int, out_bf16), dim3((unsigned)(turns < blocks ? turns : blocks)), kRowsThreads, smem, s, p) != cudaSuccess)
        return ABS_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? ABS_OK : ABS_ERR_CUDA;
}

static abs_status_t matmul_impl(abs_fmt_t fmt, const void* a_codes, const void* a_scales, const float* a_alpha, const void* b_codes,
                                const void* b_scales, const float* b_alpha, int64_t m, int64_t n, int64_t k, void* c_f32,
                                void* workspace, size_t workspace_bytes, void* stream, int32_t stall_step, bool out_bf16 = false,
                                float* next_alpha = nullptr, float next_denom = 0.0f) {
    const absq::CallRange range("abs_matmul");
    if (fmt != ABS_FMT_IF4 && fmt != ABS_FMT_NVFP4) return ABS_ERR_FMT;
    if (!gemm_shape_ok(fmt, m, n, k)) return ABS_ERR_SHAPE;
    if (!a_codes || !a_scales || !a_alpha || !b_codes || !b_scales || !b_alpha || !c_f32 || !workspace) return ABS_ERR_NULL;
    const uintptr_t all = (uintptr_t)a_codes | (uintptr_t)a_scales | (uintptr_t)b_codes | (uintptr_t)b_scales | (uintptr_t)c_f32;
    if ((all & 15u) || ((uintptr_t)workspace & 1023u)) return ABS_ERR_ALIGN;
    if (workspace_bytes < abs_matmul_workspace_bytes(fmt, m, n, k)) return ABS_ERR_SIZE;
    const GemmLayout L = gemm_layout(fmt, m, n, k);
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t* ws = (uint8_t*)workspace;
    const bool has_int = fmt == ABS_FMT_IF4;
    // the opt-in to more than 48 KiB of dynamic shared memory is per device
    static std::once_flag attr_once[64];
    static cudaError_t attr_err[64];
    static int sm_count[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return ABS_ERR_CUDA;
    std::call_once(attr_once[dev], [dev]() {
        if (cudaDeviceGetAttribute(&sm_count[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sm_count[dev] < 1)
            sm_count[dev] = 1;
        attr_err[dev] = cudaSuccess;
#define ABS_GEMM_ATTR(P, O, B)                                                                                         \
    if (attr_err[dev] == cudaSuccess)                                                                                   \
        attr_err[dev] = cudaFuncSetAttribute(if4_gemm_kernel<P, O, B>, cudaFuncAttributeMaxDynamicSharedMemorySize,      \
                                             kGemmSmemBytes<P, B>)
        ABS_GEMM_ATTR(2, false, 1); ABS_GEMM_ATTR(2, true, 1);
        ABS_GEMM_ATTR(1, false, 1); ABS_GEMM_ATTR(1, true, 1);
        ABS_GEMM_ATTR(1, false, 2); ABS_GEMM_ATTR(1, true, 2);
#undef ABS_GEMM_ATTR
        if (attr_err[dev] == cudaSuccess)
            attr_err[dev] = cudaFuncSetAttribute(nvfp4_pair_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmemBytes);
        if (attr_err[dev] == cudaSuccess)
            attr_err[dev] = cudaFuncSetAttribute(nvfp4_pair_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmemBytes);
        if (attr_err[dev] == cudaSuccess)
            attr_err[dev] = cudaFuncSetAttribute(skinny_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSkinnySmemBytes);
        if (attr_err[dev] == cudaSuccess)
            attr_err[dev] = cudaFuncSetAttribute(skinny_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSkinnySmemBytes);
        for (int i = 0; i < 16; ++i)
            if (attr_err[dev] == cudaSuccess)
                attr_err[dev] = cudaFuncSetAttribute(rows_kernel_of(1 << (i >> 2), i & 1, i & 2), cudaFuncAttributeMaxDynamicSharedMemorySize, kRowsMaxSmem);
    });
    if (attr_err[dev] != cudaSuccess) return ABS_ERR_CUDA;
    // (the self-test of the waits is for kernels that have some)
    if (stall_step < 0 && rows_rule(fmt, m, n, k, sm_count[dev]))
        return rows_matmul(has_int, a_codes, a_scales, a_alpha, b_codes, b_scales, b_alpha, m, n, k, c_f32, ws, s, sm_count[dev], out_bf16,
                           next_alpha, next_denom);
    SkinnyPlan P;
    if (skinny_plan(fmt, m, n, k, sm_count[dev] < kMaxSms ? sm_count[dev] : kMaxSms, P))
        return skinny_matmul(P, a_codes, a_scales, a_alpha, b_codes, b_scales, b_alpha, m, n, k, c_f32, ws, s, stall_step, out_bf16,
                             next_alpha, next_denom);

    GemmMaps<1> maps1;
    GemmMaps<2> maps2;
    if (has_int) {
        for (int p = 0; p < 2; ++p)
            if (!plane_map(&maps2.a[p], ws + L.off_a + p * L.plane_a, (uint64_t)m, (uint64_t)k / 2) ||
                !plane_map(&maps2.b[p], ws + L.off_b + p * L.plane_b, (uint64_t)n, (uint64_t)k / 2))
                return ABS_ERR_CUDA;
        if (!scale_map(&maps2.sa, const_cast<void*>(a_scales), (uint64_t)m, (uint64_t)k / 16) ||
            !scale_map(&maps2.sb, const_cast<void*>(b_scales), (uint64_t)n, (uint64_t)k / 16))
            return ABS_ERR_CUDA;
        SplitOperand so[2];
        for (int op = 0; op < 2; ++op) {
            const size_t off = op ? L.off_b : L.off_a, plane = op ? L.plane_b : L.plane_a;
            so[op].codes = (const uint4*)(op ? b_codes : a_codes);
            so[op].scales = (const uint8_t*)(op ? b_scales : a_scales);
            so[op].plane_h = (uint4*)(ws + off);
            so[op].plane_l = (uint4*)(ws + off + plane);
            so[op].pairs = (op ? n : m) * (k / 32);
        }
        int64_t blocks = (so[0].pairs + so[1].pairs + 255) / 256;
        if (blocks > 148 * 8) blocks = 148 * 8;
        if (launch_pdl(if4_split_kernel, dim3((unsigned)blocks), 256, 0, s, so[0], so[1], (int*)ws) != cudaSuccess) return ABS_ERR_CUDA;
    } else {
        if (!plane_map(&maps1.a[0], const_cast<void*>(a_codes), (uint64_t)m, (uint64_t)k / 2) ||
            !plane_map(&maps1.b[0], const_cast<void*>(b_codes), (uint64_t)n, (uint64_t)k / 2))
            return ABS_ERR_CUDA;
        maps1.sfa = ws + L.off_a;
        maps1.sfb = ws + L.off_b;
        TileOperand to[2];
        for (int op = 0; op < 2; ++op) {
            to[op].scales = (const uint8_t*)(op ? b_scales : a_scales);
            to[op].tiled = ws + (op ? L.off_b : L.off_a);
            to[op].rows = op ? n : m;
            to[op].items = (to[op].rows + 127) / 128 * (k / kStageK) * 32;
            to[op].pitch = (uint32_t)(k / 16);
            to[op].ksteps = (uint32_t)(k / kStageK);
        }
        int64_t blocks = (to[0].items + to[1].items + 255) / 256;
        if (blocks > 148 * 8) blocks = 148 * 8;
        if (launch_pdl(sf_tile_kernel, dim3((unsigned)blocks), 256, 0, s, to[0], to[1], (int*)ws) != cudaSuccess) return ABS_ERR_CUDA;
    }
    const int32_t tiles_m = (int32_t)((m + kTileM - 1) / kTileM), tiles_n = (int32_t)(n / kTileN);
    const int64_t num_tiles = (int64_t)tiles_m * tiles_n;
    const dim3 pgrid((unsigned)(num_tiles < sm_count[dev] ? num_tiles : sm_count[dev]));
    cudaError_t e;
#define ABS_LAUNCH_GEMM(P, O, B)                                                                                        \
    e = launch_pdl(if4_gemm_kernel<P, O, B>, pgrid, kGemmThreads<P>, kGemmSmemBytes<P, B>, s, maps##P, a_alpha, b_alpha, c_f32, tiles_m, tiles_n, \
                   (int32_t)(k / (kStageK * B)), (int32_t)m, (int*)ws, stall_step, next_alpha, next_denom)
    if (!has_int && pair_rule(out_bf16, tiles_m, tiles_n, k, sm_count[dev])) {
        e = launch_pdl(out_bf16 ? nvfp4_pair_kernel<true> : nvfp4_pair_kernel<false>, dim3((unsigned)sm_count[dev]), kPairThreads, kPairSmemBytes, s, maps1,
                       a_alpha, b_alpha, c_f32, tiles_m, tiles_n, (int32_t)(k / kStageK), (int32_t)m, (int*)ws, stall_step, next_alpha, next_denom);
        return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? ABS_OK : ABS_ERR_CUDA;
    }
    const bool long_steps = !has_int && k % (2 * kStageK) == 0;      // NVFP4: K-steps of 512 where K allows
    if (has_int && out_bf16) ABS_LAUNCH_GEMM(2, true, 1);
    else if (has_int) ABS_LAUNCH_GEMM(2, false, 1);
    else if (long_steps && out_bf16) ABS_LAUNCH_GEMM(1, true, 2);
    else if (long_steps) ABS_LAUNCH_GEMM(1, false, 2);
    else if (out_bf16) ABS_LAUNCH_GEMM(1, true, 1);
    else ABS_LAUNCH_GEMM(1, false, 1);
#undef ABS_LAUNCH_GEMM
    if (e != cudaSuccess) return ABS_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? ABS_OK : ABS_ERR_CUDA;
}

abs_status_t abs_matmul(abs_fmt_t fmt, const void* a_codes, const void* a_scales, const float* a_alpha, const void* b_codes,
                        const void* b_scales, const float* b_alpha, int64_t m, int64_t n, int64_t k, float* c_f32,
                        void* workspace, size_t workspace_bytes, void* stream) {
    return matmul_impl(fmt, a_codes, a_scales, a_alpha, b_codes, b_scales, b_alpha, m, n, k, c_f32, workspace, workspace_bytes, stream, -1);
}

abs_status_t abs_matmul_bf16(abs_fmt_t fmt, const void* a_codes, const void* a_scales, const float* a_alpha, const void* b_codes,
                             const void* b_scales, const float* b_alpha, int64_t m, int64_t n, int64_t k, void* c_bf16,
                             void* workspace, size_t workspace_bytes, void* stream) {
    return matmul_impl(fmt, a_codes, a_scales, a_alpha, b_codes, b_scales, b_alpha, m, n, k, c_bf16, workspace, workspace_bytes, stream, -1,
                       true);
}

static abs_status_t matmul_scaled(abs_fmt_t fmt, const void* a_codes, const void* a_scales, const float* a_alpha, const void* b_codes,
                                  const void* b_scales, const float* b_alpha, int64_t m, int64_t n, int64_t k, void* c_bf16, abs_fmt_t next_fmt,
                                  float* next_alpha, void* workspace, size_t workspace_bytes, void* stream, int32_t stall_step) {
    if (!next_alpha) return ABS_ERR_NULL;
    float m_fp;
    switch (next_fmt) {
        case ABS_FMT_NVFP4: case ABS_FMT_IF4: case ABS_FMT_IF4_BS8: case ABS_FMT_NVFP4_BS8: m_fp = 6.0f; break;
        case ABS_FMT_IF3: case ABS_FMT_IF3_BS8: m_fp = 4.0f; break;
        case ABS_FMT_IF6_E2M3: m_fp = 7.5f; break;
        case ABS_FMT_IF6_E3M2: m_fp = 28.0f; break;
        default: return ABS_ERR_FMT;
    }
    return matmul_impl(fmt, a_codes, a_scales, a_alpha, b_codes, b_scales, b_alpha, m, n, k, c_bf16, workspace, workspace_bytes, stream, stall_step,
                       true, next_alpha, m_fp * 448.0f);
}

abs_status_t abs_matmul_bf16_scaled(abs_fmt_t fmt, const void* a_codes, const void* a_scales, const float* a_alpha,
                                    const void* b_codes, const void* b_scales, const float* b_alpha, int64_t m, int64_t n, int64_t k,
                                    void* c_bf16, abs_fmt_t next_fmt, float* next_alpha, void* workspace, size_t workspace_bytes,
                                    void* stream) {
    return matmul_scaled(fmt, a_codes, a_scales, a_alpha, b_codes, b_scales, b_alpha, m, n, k, c_bf16, next_fmt, next_alpha, workspace,
                         workspace_bytes, stream, -1);
}

abs_status_t abs_selftest_matmul_stall(abs_fmt_t fmt, const void* a_codes, const void* a_scales, const float* a_alpha,
                                       const void* b_codes, const void* b_scales, const float* b_alpha, int64_t m, int64_t n,
                                       int64_t k, float* c_f32, void* workspace, size_t workspace_bytes, void* stream,
                                       int32_t stall_step) {
    if (stall_step < 0) return ABS_ERR_SHAPE;
    return matmul_impl(fmt, a_codes, a_scales, a_alpha, b_codes, b_scales, b_alpha, m, n, k, c_f32, workspace, workspace_bytes, stream,
                       stall_step);
}

abs_status_t abs_selftest_matmul_stall_scaled(abs_fmt_t fmt, const void* a_codes, const void* a_scales, const float* a_alpha,
                                              const void* b_codes, const void* b_scales, const float* b_alpha, int64_t m, int64_t n,
                                              int64_t k, void* c_bf16, abs_fmt_t next_fmt, float* next_alpha, void* workspace,
                                              size_t workspace_bytes, void* stream, int32_t stall_step) {
    if (stall_step < 0) return ABS_ERR_SHAPE;
    return matmul_scaled(fmt, a_codes, a_scales, a_alpha, b_codes, b_scales, b_alpha, m, n, k, c_bf16, next_fmt, next_alpha, workspace,
                         workspace_bytes, stream, stall_step);
}

abs_status_t abs_matmul_check(const void* workspace, void* stream) {
    if (!workspace) return ABS_ERR_NULL;
    int word = 0;
    if (cudaMemcpyAsync(&word, workspace, sizeof(int), cudaMemcpyDeviceToHost, (cudaStream_t)stream) != cudaSuccess ||
        cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess)
        return ABS_ERR_CUDA;
    return word == 0 ? ABS_OK : ABS_ERR_CUDA;
}

}  // extern "C"
