// The NVFP4 product with many tiles: as if4_gemm_kernel<1> (abs_gemm.cu), but a block takes two neighbouring 128 x 128 tiles of C at a time.
//
// What bounds large NVFP4 products is power, and what the tensor cores themselves do not spend goes into bringing operands from the L2: a 128 x 128
// tile brings two boxes of codes per MMA.  Two tiles that share their box of A bring one and a half, and read A once for two MMAs (collector buffer).
// Three accumulators of 128 columns are used in turn, so that the epilogue of one pair of tiles runs under the MMAs of the next: the first tile
// of the next pair finds a free accumulator, the second waits until the first one of the pair before is in the epilogue's registers, and meanwhile
// the first tile's MMAs run up to kLead steps ahead.  Tensor memory: 3 x 128 columns of accumulators, two slots of 48 columns of scales.
// Pipeline: four stages of K = 256 (48 KB: A, B, B), the scales of a step in a ring of four (2 KB of the 128x4 tiles of sf_tile_kernel for each of A, B, B,
// one bulk copy each, by a thread of their own: 1 - 2 %).  Four warps copy them into tensor memory; a stage's `full` barrier counts its loads and these
// warps, its `empty` barrier frees its shared memory and its slot of scales.  A step, eight MMAs of 64 cycles, takes some 750 cycles (1130 for eight MMAs in
// if4_gemm_kernel<1>); waiting for the next step's operands before the last MMAs of a step, as the IF4 loop does, made it 10 % slower: with two slots
// the next step's scales come after the MMAs of the step before.
// The epilogue stores as in if4_gemm_kernel (turned through shared memory for whole lines, bf16 products took 2 - 18 % longer, most with a short K).
// 1000 x 14336 x 4096, bf16, 41.9 -> 36.3 us, 2048 x 4096 x 4096 27.4 -> 23.5, 4096^3 42.0 -> 36.2; at the power cap 8192 x 14336 x 4096 321 -> 274 (FP32 388 -> 326),
// 2048 x 8192 x 14336 161 -> 132.  The results are those of if4_gemm_kernel<1>, bit for bit.
#pragma once
#include "abs_tc.cuh"

#include <type_traits>

namespace absq {

constexpr int kPairStages = 4, kPairStageBytes = 3 * kPlaneBytes, kPairScaleBufs = 4, kPairScaleBytes = 128 * (kStageK / 16);
constexpr int kPairAccBufs = 3, kPairSlots = 2, kPairLead = 2;
constexpr int kPairThreads = 32 * (2 + 4 + 4 + 1);
constexpr int kPairSmemBytes = kPairStages * kPairStageBytes + kPairScaleBufs * 3 * kPairScaleBytes + 1024 /* alignment slack */ + 512 /* barriers */;

// The pairs of tiles of a block: in `rounds` full rounds of the grid a pair each, then, where the rest is at most half a round, single tiles.
struct PairWalk {
    int32_t tiles_m, tiles_n, pairs_n, pairs, rounds;
    bool single_rest;
    __device__ __forceinline__ PairWalk(int32_t tm, int32_t tn) : tiles_m(tm), tiles_n(tn), pairs_n((tn + 1) / 2) {
        pairs = tiles_m * pairs_n;
        rounds = pairs / (int32_t)gridDim.x;
        single_rest = 2 * (pairs - rounds * (int32_t)gridDim.x) <= (int32_t)gridDim.x;
    }
    // Task i of this block: tile row, first tile column, number of tiles; false when there is none.
    __device__ __forceinline__ bool task(int32_t i, int32_t& tile_m, int32_t& tile_n, int32_t& width) const {
        if (i > rounds) return false;
        const bool single = single_rest && i == rounds;
        const int32_t b = (int32_t)blockIdx.x, p = i * (int32_t)gridDim.x + (single ? b >> 1 : b);
        if (p >= pairs) return false;
        int32_t pn;
        tile_of(p, tiles_m, pairs_n, tile_m, pn);
        tile_n = 2 * pn + (single ? b & 1 : 0);
        width = min(single ? 1 : 2, tiles_n - tile_n);
        return width > 0;
    }
};

// OUT_BF16, error, stall_step, next_alpha: as in if4_gemm_kernel.
template <bool OUT_BF16>
__global__ void __launch_bounds__(kPairThreads, 1)
nvfp4_pair_kernel(const __grid_constant__ GemmMaps<1> maps, const float* __restrict__ alpha_a, const float* __restrict__ alpha_b,
                  void* __restrict__ c_out, int32_t tiles_m, int32_t tiles_n, int32_t k_iters, int32_t m_rows, int* __restrict__ error,
                  int32_t stall_step, float* __restrict__ next_alpha, float next_denom) {
    constexpr int kBlocks = kStageK / kMmaK;                          // MMA K-blocks of a step
    constexpr uint32_t kSfBase = kPairAccBufs * kTileN, kSlotCols = 3 * 4 * kBlocks, kTmemCols = 512;
    static_assert(kSfBase + kPairSlots * kSlotCols <= kTmemCols, "tensor memory");
    extern __shared__ uint8_t pair_smem_raw[];
    const uint32_t raw = smem_u32(pair_smem_raw), base = (raw + 1023u) & ~1023u;
    const uint32_t sf0 = base + kPairStages * kPairStageBytes, bars = sf0 + kPairScaleBufs * 3 * kPairScaleBytes;
    const uint32_t full0 = bars, empty0 = bars + 64, sf_full0 = bars + 128, sf_empty0 = bars + 192, acc_full0 = bars + 256, acc_empty0 = bars + 320;
    const uint32_t drained = bars + 384;
    uint32_t* tmem_word = reinterpret_cast<uint32_t*>(pair_smem_raw + (bars - raw) + 448);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        for (int s = 0; s < kPairStages; ++s) { mbar_init(full0 + 8 * s, 1 + 4); mbar_init(empty0 + 8 * s, 1); }
        for (int i = 0; i < kPairScaleBufs; ++i) { mbar_init(sf_full0 + 8 * i, 1); mbar_init(sf_empty0 + 8 * i, 4); }
        for (int i = 0; i < kPairAccBufs; ++i) { mbar_init(acc_full0 + 8 * i, 1); mbar_init(acc_empty0 + 8 * i, 4); }
        mbar_init(drained, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) { tmem_alloc(smem_u32(tmem_word), kTmemCols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, *tmem_word, 0);
    const PairWalk walk(tiles_m, tiles_n);
    int32_t tile_m, tile_n, width;
    pdl_wait();

    if (warp == 0) {
        if (lane == 0) {
            // ---- codes
            uint32_t it = 0, s = 0;                                   // step and its stage
            bool ok = true;
            for (int32_t i = 0; ok && walk.task(i, tile_m, tile_n, width); ++i) {
                for (int32_t kt = 0; kt < k_iters; ++kt, ++it) {
                    if (!mbar_wait(empty0 + 8 * s, ((it / kPairStages) & 1u) ^ 1u)) { atomicExch(error, 1); ok = false; break; }
                    const uint32_t st = base + s * kPairStageBytes, bar = full0 + 8 * s;
                    mbar_expect_tx(bar, (1 + width) * kPlaneBytes);
                    if ((int32_t)it != stall_step) {                  // self-test only: the bytes announced never arrive
                        const int32_t x = kt * (kStageK / 2);
                        tma_load_2d(st, &maps.a[0], x, tile_m * kTileM, bar);
                        tma_load_2d(st + kPlaneBytes, &maps.b[0], x, tile_n * kTileN, bar);
                        if (width == 2) tma_load_2d(st + 2 * kPlaneBytes, &maps.b[0], x, (tile_n + 1) * kTileN, bar);
                    }
                    s = s + 1 == kPairStages ? 0u : s + 1;
                }
            }
        }
    } else if (warp == 10) {
        if (lane == 0) {
            // ---- scales: 2 KB per operand and step (a thread of its own: six copies a step kept one busy for 640 cycles, the MMAs take 512)
            uint32_t it = 0, b = 0;
            bool ok = true;
            for (int32_t i = 0; ok && walk.task(i, tile_m, tile_n, width); ++i) {
                const uint8_t* sfa = maps.sfa + (size_t)tile_m * k_iters * kPairScaleBytes;
                const uint8_t* sfb = maps.sfb + (size_t)tile_n * k_iters * kPairScaleBytes;
                const uint8_t* sfb1 = sfb + (size_t)k_iters * kPairScaleBytes;
                for (int32_t kt = 0; kt < k_iters; ++kt, ++it) {
                    const uint32_t at = sf0 + b * 3 * kPairScaleBytes, bar = sf_full0 + 8 * b;
                    const size_t from = (size_t)kt * kPairScaleBytes;
                    if (!mbar_wait(sf_empty0 + 8 * b, ((it / kPairScaleBufs) & 1u) ^ 1u)) { atomicExch(error, 7); ok = false; break; }
                    mbar_expect_tx(bar, (1 + width) * kPairScaleBytes);
                    if ((int32_t)it != stall_step) {
                        bulk_load(at, sfa + from, kPairScaleBytes, bar);
                        bulk_load(at + kPairScaleBytes, sfb + from, kPairScaleBytes, bar);
                        if (width == 2) bulk_load(at + 2 * kPairScaleBytes, sfb1 + from, kPairScaleBytes, bar);
                    }
                    b = b + 1 == kPairScaleBufs ? 0u : b + 1;
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMAs
            const uint64_t desc0 = operand_desc(base);
            constexpr uint64_t kPlane = kPlaneBytes >> 4;
            uint32_t s = 0, parity = 0, slot = 0, buf = 0, uses = 0;  // stage and its parity, slot of scales; next accumulator, tiles handed to accumulators so far
            bool ok = true;
            // the accumulators in turn: the n-th tile of this block uses buffer n % 3 for the (n / 3)-th time
            auto acquire = [&]() { return mbar_wait(acc_empty0 + 8 * buf, ((uses / kPairAccBufs) & 1u) ^ 1u); };
            auto advance = [&]() { ++uses; buf = buf + 1 == kPairAccBufs ? 0u : buf + 1; };
            for (int32_t i = 0; ok && walk.task(i, tile_m, tile_n, width); ++i) {
                if (!acquire()) { atomicExch(error, 4); ok = false; break; }
                const uint32_t acc0 = tmem + buf * kTileN, done0 = acc_full0 + 8 * buf;
                advance();
                uint32_t acc1 = acc0, done1 = done0;
                // K-block kb of the step in stage s, tile 0 or 1 of the pair
                auto mma = [&](auto usage, uint32_t st, uint32_t sl, int kb, uint32_t half, bool first) __attribute__((always_inline)) {
                    const uint64_t a = desc0 + (uint64_t)st * (kPairStageBytes >> 4) + ((kb * (kMmaK / 2)) >> 4);
                    const uint32_t fa = tmem + kSfBase + sl * kSlotCols + 4 * kb;
                    tc_mma_nvf4<decltype(usage)::value>(half ? acc1 : acc0, a, a + (1 + half) * kPlane, kInstrDesc, kb > 0 || !first, fa,
                                                        fa + (1 + half) * 4 * kBlocks);
                };
                using Keep = std::integral_constant<Collector, kFill>;
                using Last = std::integral_constant<Collector, kLastUse>;
                using Once = std::integral_constant<Collector, kDiscard>;
                int32_t kt = 0;
                if (width == 2) {
                    // the first tile's MMAs of up to kPairLead steps, while the second one's accumulator is emptied
                    const int32_t lead = min(kPairLead, k_iters);
                    uint32_t s1 = s, p1 = parity, sl1 = slot;
                    for (int32_t q = 0; q < lead && ok; ++q) {
                        if (!mbar_wait(full0 + 8 * s1, p1)) { atomicExch(error, 2); ok = false; break; }
                        tc_fence_after();
#pragma unroll
                        for (int kb = 0; kb < kBlocks; ++kb) mma(Once{}, s1, sl1, kb, 0, q == 0);
                        if (++s1 == kPairStages) { s1 = 0; p1 ^= 1u; }
                        sl1 ^= 1u;
                    }
                    if (!ok) break;
                    if (!acquire()) { atomicExch(error, 4); ok = false; break; }
                    tc_fence_after();
                    acc1 = tmem + buf * kTileN;
                    done1 = acc_full0 + 8 * buf;
                    advance();
                    for (; kt < lead; ++kt) {
#pragma unroll
                        for (int kb = 0; kb < kBlocks; ++kb) mma(Once{}, s, slot, kb, 1, kt == 0);
                        tc_commit(empty0 + 8 * s);
                        if (++s == kPairStages) { s = 0; parity ^= 1u; }
                        slot ^= 1u;
                    }
                }
                for (; kt < k_iters; ++kt) {
                    if (!mbar_wait(full0 + 8 * s, parity)) { atomicExch(error, 2); ok = false; break; }
                    tc_fence_after();
                    if (width == 2) {
#pragma unroll
                        for (int kb = 0; kb < kBlocks; ++kb) { mma(Keep{}, s, slot, kb, 0, false); mma(Last{}, s, slot, kb, 1, false); }
                    } else {
#pragma unroll
                        for (int kb = 0; kb < kBlocks; ++kb) mma(Once{}, s, slot, kb, 0, kt == 0);
                    }
                    tc_commit(empty0 + 8 * s);                        // the stage's shared memory and scales are free once these MMAs have run
                    if (++s == kPairStages) { s = 0; parity ^= 1u; }
                    slot ^= 1u;
                }
                if (!ok) break;
                tc_commit(done0);                                     // and the accumulators of the pair are complete
                if (width == 2) tc_commit(done1);
            }
            // All MMAs are over before the block frees its tensor memory, also where the epilogue has given up and waits for none of them.
            tc_commit(drained);
            if (!mbar_wait(drained, 0)) atomicExch(error, 8);
        }
    } else if (warp >= 6) {
        // ---- scales: this warp's copy of every step's scales, from shared memory into tensor memory
        const uint32_t lane_base = tmem + kSfBase + ((uint32_t)((warp & 3) * 32) << 16);
        uint32_t it = 0, b = 0;
        bool ok = true;
        for (int32_t i = 0; ok && walk.task(i, tile_m, tile_n, width); ++i) {
            for (int32_t kt = 0; kt < k_iters; ++kt, ++it) {
                ok = mbar_wait_warp(sf_full0 + 8 * b, (it / kPairScaleBufs) & 1u);
                uint4 r[3][kBlocks];
                if (ok) {
                    const uint4* at = reinterpret_cast<const uint4*>(pair_smem_raw + (sf0 - raw) + b * 3 * kPairScaleBytes) + lane;
#pragma unroll
                    for (int op = 0; op < 3; ++op)
#pragma unroll
                        for (int kb = 0; kb < kBlocks; ++kb)
                            if (op < 2 || width == 2) r[op][kb] = at[op * (kPairScaleBytes / 16) + kb * 32];
                    // the slot is free when the MMAs of the step before the last have run, whose stage their commit empties
                    if (it >= kPairSlots) ok = mbar_wait_warp(empty0 + 8 * ((it - kPairSlots) % kPairStages), ((it - kPairSlots) / kPairStages) & 1u);
                }
                if (!ok) { if (lane == 0) atomicExch(error, 6); break; }
                tc_fence_after();
                const uint32_t to = lane_base + (it % kPairSlots) * kSlotCols;
                tmem_store16(to, r[0][0], r[0][1], r[0][2], r[0][3]);
                tmem_store16(to + 4 * kBlocks, r[1][0], r[1][1], r[1][2], r[1][3]);
                if (width == 2) tmem_store16(to + 8 * kBlocks, r[2][0], r[2][1], r[2][2], r[2][3]);
                tmem_store_wait();
                tc_fence_before();
                __syncwarp();
                // the buffer is handed back once its values are in tensor memory: an arrive right behind the loads let the next copy overtake them
                if (lane == 0) { mbar_arrive(full0 + 8 * (it % kPairStages)); mbar_arrive(sf_empty0 + 8 * b); }
                b = b + 1 == kPairScaleBufs ? 0u : b + 1;
            }
        }
    } else {
        // ---- epilogue: this warp owns the accumulator lanes (rows of the tile) 32 (w % 4) .. 32 (w % 4) + 31
        const int quarter = warp & 3;
        const int32_t n_cols = tiles_n * kTileN;
        const float scale = __fmul_rn(__ldg(alpha_a), __ldg(alpha_b));
        const bool out_aligned32 = (reinterpret_cast<uintptr_t>(c_out) & 31u) == 0;
        uint32_t buf = 0, out_max = 0u;         // bf16 output with next_alpha: largest |C| bit pattern this thread has written
        bool all_tiles = true;
        uint32_t uses = 0;
        for (int32_t i = 0; all_tiles && walk.task(i, tile_m, tile_n, width); ++i) {
            const bool own_row_valid = tile_m * kTileM + quarter * 32 + lane < m_rows;   // the row whose values this thread holds
            const size_t row = (size_t)(tile_m * kTileM + quarter * 32 + lane) * (size_t)n_cols;
            for (int32_t half = 0; half < width; ++half, ++uses) {
                all_tiles = mbar_wait_warp(acc_full0 + 8 * buf, (uses / kPairAccBufs) & 1u);
                if (!all_tiles) { if (lane == 0) atomicExch(error, 3); break; }
                tc_fence_after();
                const uint32_t lane_base = tmem + buf * kTileN + ((uint32_t)(quarter * 32) << 16);
                const size_t first = row + (size_t)(tile_n + half) * kTileN;
                // (one copy of the loop for either alignment: with the choice inside it aligned bf16 products took 1 - 2 % longer)
                const auto columns = [&](auto whole) __attribute__((always_inline)) {
                    uint4 held = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                    for (int chunk = 0; chunk < kTileN / 32; ++chunk) {
                        uint32_t r[32];
                        tmem_load32(lane_base + chunk * 32, r);
                        tmem_load_wait();
                        if (chunk == kTileN / 32 - 1) {                    // everything is in registers: the accumulator's next tile may start
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(acc_empty0 + 8 * buf);
                        }
                        float v[32];
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(r[e]);
                        if (own_row_valid) {                               // the last row block may be partial
#pragma unroll
                            for (int q = 0; q < 2; ++q)
                                store_columns16<OUT_BF16, decltype(whole)::value>(c_out, first + chunk * 32 + 16 * q, v + 16 * q, scale, chunk + q == 0,
                                                                                  chunk == kTileN / 32 - 1 && q == 1, held, next_alpha != nullptr, out_max);
                        }
                    }
                };
                if (out_aligned32) columns(std::true_type{});
                else columns(std::false_type{});
                buf = buf + 1 == kPairAccBufs ? 0u : buf + 1;
            }
        }
        // The global maximum of |C| as written (bf16): as in if4_gemm_kernel.
        if (OUT_BF16 && next_alpha != nullptr && all_tiles) {
            const uint32_t wmax = __reduce_max_sync(0xFFFFFFFFu, max(out_max & 0xFFFFu, out_max >> 16));
            if (lane == 0) {
                atomicMax(reinterpret_cast<unsigned int*>(error) + 1, wmax);
                __threadfence();
                const int ticket = atomicAdd(error + 2, 1);
                if (ticket == (int)gridDim.x * 4 - 1) {
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
