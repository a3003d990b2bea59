// Transposed group-quantize kernel for the 4-bit formats (IF4, NVFP4): groups run down the columns of the
// row-major input (Sec. 4.1: both operands of the weight-gradient product are quantized along the token
// dimension), with the Hadamard and stochastic-rounding options of the gradient path.
#pragma once
#include "abs_opt4.cuh"
#include <type_traits>

namespace absq {

// ----------------------------------------------------------------------------- transposed quantize

// Quantizes the TRANSPOSE of a row-major [rows, cols] matrix without materialising it: groups are 16
// consecutive ROWS of one column (Sec. 4.1: both operands of the weight-gradient product are quantized
// along the token dimension).  Output = what the plain kernel would give for the [cols, rows] matrix:
// codes_t [cols, rows/2 bytes], scales_t [cols, rows/16].
// Blocks of 128 threads walk over tiles of 64 rows x 128 columns.  A tile is brought into shared memory with
// 16-byte asynchronous copies (cp.async), double buffered: the copies of the block's next tile are in
// flight while it encodes the current one.  Thread c reads its column's values down the tile and encodes
// the four groups of 16 rows; those are neighbours in the transposed output, so their codes leave as one
// 256-bit store and their scale bytes as one 32-bit store whenever the tile is complete and the output
// addresses allow it.
constexpr int kTransUnroll = 4;
constexpr int kTransTileCols = 128;                                                 // one thread per column
constexpr int kTransTileRowBlocks = 4;
constexpr int kTransRowChunks = kTransTileCols / 8, kTransRowLines = kTransTileCols / 64;   // 16-byte chunks, 128-byte lines of a row
constexpr int kTransStageElems = 16 * kTransTileRowBlocks * kTransTileCols;        // bf16 elements per stage
constexpr int kTransSmemBytes = 2 * kTransStageElems * 2;                           // two stages: 32 KB, which needs no attribute
static_assert(kTransSmemBytes <= 48 * 1024 - 64, "dynamic shared memory without an attribute");

// Blocks per SM the kernels are compiled for (shared memory would allow six).  What bounds them is the arithmetic pipes, so what helps is that another block
// runs while one waits at a barrier or for its tile: blocks of 128 threads and columns instead of 256 (three per SM; with stochastic rounding two).
// us, kernel alone, 256 / 128 columns, 8192 x 14336, 4096 x 4096 and 2048 x 2048: IF4 67.7 / 62.7, 11.9 / 11.4, 5.9 / 5.5; Hadamard 85.5 / 80.5, 14.7 / 13.8,
// 7.0 / 6.2; Hadamard and SR 142.5 / 140.0, 25.3 / 22.4, 10.6 / 9.4; as the emulation pass 199 / 195, 34.7 / 30.6, 10.2 / 10.2; NVFP4 52.8 / 46.8, 8.2 / 8.0,
// 4.2 / 4.2.  64 columns: equal or slower.  Six against five blocks: IF4 with Hadamard 1 to 10 % slower (fewer registers), the others up to 4 % faster where tiles abound;
// SR with five against four: 2 to 5 % faster from 2048 x 4096 up, but the emulation pass of 2048 x 2048 18 % slower.
constexpr int trans_blocks_per_sm(bool has_int, bool rht, bool sr, bool emul) { return sr ? (emul ? 4 : 5) : has_int && rht ? 5 : 6; }

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all_but_one() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// 16-point transform of one group held as sixteen floats: sign flips, the h = 1 stage with scalar adds,
// the h = 2, 4, 8 stages on register pairs with packed add / fused subtract, times 1/4 (same arithmetic as
// hadamard16, every result rounded to FP32 once).
__device__ __forceinline__ void hadamard16_pairs(float (&x)[16], uint32_t sign_mask) {
    uint64_t P[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float p = __uint_as_float(__float_as_uint(x[2 * i]) ^ (((sign_mask >> (2 * i)) & 1u) << 31));
        const float q = __uint_as_float(__float_as_uint(x[2 * i + 1]) ^ (((sign_mask >> (2 * i + 1)) & 1u) << 31));
        P[i] = pack2(__fadd_rn(p, q), __fsub_rn(p, q));
    }
    const uint64_t NEG1 = pack2(-1.0f, -1.0f), QUARTER = pack2(0.25f, 0.25f);
#pragma unroll
    for (int h = 1; h < 8; h <<= 1) {
#pragma unroll
        for (int base = 0; base < 8; base += 2 * h) {
#pragma unroll
            for (int j = base; j < base + h; ++j) {
                const uint64_t p = P[j], q = P[j + h];
                P[j] = add2(p, q);
                P[j + h] = fma2(q, NEG1, p);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) unpack2(mul2(P[i], QUARTER), x[2 * i], x[2 * i + 1]);
}

// SR: stochastic rounding of both candidates (App. B); element indices, and so the Philox counters, are
// those of the transposed matrix.  scale_mul is 17/16 with that option and 1 otherwise.
// EMUL: the emulation pass of Sec. 4.1 along the columns.  Every group is decoded from the
// registers that hold its codes and written back over its own input values in the shared-memory tile; the
// finished tile then leaves with coalesced 16-byte stores to `out`, a [rows, cols] matrix in the ORIGINAL
// orientation.  Codes and scales (transposed layout) are stored only when `store_codes` is set.
template <bool HAS_INT, bool FROM_SLOT, bool RHT, bool SR, bool EMUL>
__global__ void __launch_bounds__(kTransTileCols, trans_blocks_per_sm(HAS_INT, RHT, SR, EMUL))
quantize4_transposed_kernel(const uint16_t* __restrict__ in, uint2* __restrict__ codes_t, uint8_t* __restrict__ scales_t, const AlphaSrc alpha_src,
                            int64_t rows, int64_t cols, uint32_t sign_mask, float scale_mul, const PhiloxKeys keys, uint64_t ctr_base,
                            uint16_t* __restrict__ out, bool store_codes) {
    extern __shared__ __align__(16) uint16_t trans_smem[];
    pdl_launch_dependents();
    const int64_t rblocks = rows / 16;
    const int64_t ntx = (cols + kTransTileCols - 1) / kTransTileCols;
    const int64_t nty = (rblocks + kTransTileRowBlocks - 1) / kTransTileRowBlocks;
    const int64_t ntiles = ntx * nty;
    // vector stores need 32-byte aligned code addresses and 4-byte aligned scale addresses for every column
    const bool vec_ok = (rblocks % kTransTileRowBlocks) == 0 &&
                        ((reinterpret_cast<uintptr_t>(codes_t) & 31u) == 0) && ((reinterpret_cast<uintptr_t>(scales_t) & 3u) == 0);

    // issue the asynchronous copies of tile t = (ty, tx) into stage s (one commit group per call, possibly empty).
    auto issue = [&](int64_t t, uint32_t ty, uint32_t tx, int s) {
        if (t < ntiles) {
            const int64_t rb0 = (int64_t)ty * kTransTileRowBlocks, c0 = (int64_t)tx * kTransTileCols;
            const int nrb = (int)min((int64_t)kTransTileRowBlocks, rblocks - rb0);
            const int ncols = (int)min((int64_t)kTransTileCols, cols - c0);
            uint16_t* stage = trans_smem + s * kTransStageElems;
            const uint16_t* src = in + rb0 * 16 * cols + c0;
            if (ncols == kTransTileCols && nrb == kTransTileRowBlocks) {
                // complete tile: chunk ch = thread + threads * j of 16 bytes lands at stage + 8 ch and comes
                // from row (thread / chunks of a row) + 8 j, columns 8 (thread % chunks of a row) ...
                uint16_t* dst = stage + 8 * threadIdx.x;
                const uint16_t* from = src + (int64_t)(threadIdx.x / kTransRowChunks) * cols + 8 * (threadIdx.x % kTransRowChunks);
                const int64_t step = 8 * cols;
#pragma unroll
                for (int j = 0; j < 2 * kTransTileRowBlocks; ++j)
                    cp_async16(dst + j * 8 * kTransTileCols, from + j * step);
            } else if (ncols == kTransTileCols) {        // full-width tile
                for (int ch = threadIdx.x; ch < 16 * nrb * kTransRowChunks; ch += blockDim.x) {
                    const int r = ch / kTransRowChunks, q = ch % kTransRowChunks;
                    cp_async16(stage + r * kTransTileCols + q * 8, src + (int64_t)r * cols + q * 8);
                }
            } else {                                     // ragged last column tile
                const int chunks_per_row = ncols / 8;
                for (int ch = threadIdx.x; ch < 16 * nrb * chunks_per_row; ch += blockDim.x) {
                    const int r = ch / chunks_per_row, q = ch - r * chunks_per_row;
                    cp_async16(stage + r * kTransTileCols + q * 8, src + (int64_t)r * cols + q * 8);
                }
            }
        }
        cp_async_commit();
    };

    int s = 0;
    // Tile counts fit 32 bits (a tile is 8192 elements).  The block's tiles are t, t + grid, ...: their
    // coordinates advance by (grid / ntx, grid % ntx) with one carry, so only the first needs a division.
    int64_t t = blockIdx.x;
    const uint32_t ntx32 = (uint32_t)ntx, step_y = gridDim.x / ntx32, step_x = gridDim.x - step_y * ntx32;
    uint32_t ty = blockIdx.x / ntx32, tx = blockIdx.x - ty * ntx32;
    {   // before the wait (see prefetch_l2): the block's first tile, a line of 128 bytes per thread
        const int64_t r = (int64_t)ty * 16 * kTransTileRowBlocks + threadIdx.x / kTransRowLines, c = (int64_t)tx * kTransTileCols + 64 * (threadIdx.x % kTransRowLines);
        if (r < rows && c < cols) prefetch_l2(in + r * cols + c);
    }
    pdl_wait();
    issue(t, ty, tx, 0);                             // its copies are on their way while alpha is read
    const float alpha = resolve_alpha<FROM_SLOT>(alpha_src);                 // T2
    const float inv_a6 = __frcp_rn(__fmul_rn(alpha, 6.0f));                  // T3
    for (; t < ntiles; t += gridDim.x, s ^= 1) {
        uint32_t ty_next = ty + step_y, tx_next = tx + step_x;
        if (tx_next >= ntx32) { tx_next -= ntx32; ++ty_next; }
        issue(t + gridDim.x, ty_next, tx_next, s ^ 1);   // prefetch the block's next tile into the other stage
        cp_async_wait_all_but_one();                 // this thread's copies of tile t have landed
        __syncthreads();                             // ... and everybody else's
        const int64_t rb0 = (int64_t)ty * kTransTileRowBlocks, c0 = (int64_t)tx * kTransTileCols;
        const int nrb = (int)min((int64_t)kTransTileRowBlocks, rblocks - rb0);
        const int ncols = (int)min((int64_t)kTransTileCols, cols - c0);
        uint16_t* stage = trans_smem + s * kTransStageElems;
        const int c = threadIdx.x;
        // FULL: a complete tile whose outputs may leave as vector stores (the usual case): no per-group
        // bounds checks.  Otherwise the ragged-tile path with the same arithmetic.
        auto encode_column = [&](auto full_tag) {
            constexpr bool FULL = decltype(full_tag)::value;
            const bool vec = FULL || vec_ok;
            uint32_t cw[2 * kTransTileRowBlocks];
            uint32_t sbytes = 0u;
#pragma unroll kTransUnroll
            for (int k = 0; k < kTransTileRowBlocks; ++k) {
                if constexpr (!FULL) {
                    if (k >= nrb) break;
                }
                float x[16];
                const uint16_t* colp = stage + 16 * k * kTransTileCols + c;
#pragma unroll
                for (int i = 0; i < 16; ++i) x[i] = __uint_as_float((uint32_t)colp[i * kTransTileCols] << 16);
                if constexpr (RHT) hadamard16_pairs(x, sign_mask);   // along the group, i.e. down the column
                const float m0 = max3abs(x[0], x[1], x[2]), m1 = max3abs(x[3], x[4], x[5]);
                const float m2 = max3abs(x[6], x[7], x[8]), m3 = max3abs(x[9], x[10], x[11]);
                const float m4 = max3abs(x[12], x[13], x[14]);
                const float gmax = fmaxf(max3abs(m0, m1, m2), max3abs(m3, m4, x[15]));   // G1
                const float tt = __fmul_rn(__fmul_rn(gmax, inv_a6), scale_mul);          // G2
                const uint32_t sb = e4m3_encode(tt);                                     // G3
                const float d = __fmul_rn(e4m3_value(sb), alpha);                        // G5
                const float r = __frcp_rn(d);
                uint32_t sbyte = 0u, c_lo = 0u, c_hi = 0u;
                const int64_t g = (c0 + c) * rblocks + rb0 + k;      // group index in the transposed matrix
                if constexpr (SR) {
                    if (sb != 0u) {
                        const uint64_t i8 = ctr_base + (uint64_t)g * 2u;   // Philox blocks 2g, 2g+1: elements 16g .. 16g+15
                        const uint4 p0 = philox4x32_10((uint32_t)i8, (uint32_t)(i8 >> 32), keys);
                        const uint4 p1 = philox4x32_10((uint32_t)i8 + 1u, (uint32_t)(i8 >> 32), keys);
                        const uint32_t rnd[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
                        encode_body4_sr<HAS_INT, true>(x, rnd, sb, d, r, sbyte, c_lo, c_hi);
                    }
                } else if ((sb - 8u) >= 118u) {
                    if (sb != 0u) encode_body4<HAS_INT, HAS_INT>(x, sb, d, r, sbyte, c_lo, c_hi);
                } else {
                    encode_body4<HAS_INT, false>(x, sb, d, r, sbyte, c_lo, c_hi);
                }
                if constexpr (EMUL) {
                    // decode the group from its codes (arithmetic of the dequantize kernel) over its own inputs
                    const bool is_int = HAS_INT && (sbyte & 0x80u);
                    const float dd = is_int ? __fmul_rn(d, __uint_as_float(0x3F5B6DB7u)) : d;
                    const float addend = is_int ? -1032.0f : -0.0f;
                    const uint64_t D2 = pack2(dd, dd);
                    uint32_t lo[4], hi[4];
                    dequant_word4<HAS_INT>(c_lo, is_int, addend, D2, lo);
                    dequant_word4<HAS_INT>(c_hi, is_int, addend, D2, hi);
                    uint16_t* colw = stage + 16 * k * kTransTileCols + c;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        colw[(2 * i) * kTransTileCols] = (uint16_t)lo[i];
                        colw[(2 * i + 1) * kTransTileCols] = (uint16_t)(lo[i] >> 16);
                        colw[(8 + 2 * i) * kTransTileCols] = (uint16_t)hi[i];
                        colw[(9 + 2 * i) * kTransTileCols] = (uint16_t)(hi[i] >> 16);
                    }
                    if (!store_codes) continue;
                }
                if (vec) {
                    // k is a runtime index: select the slot without dynamic register indexing
#pragma unroll
                    for (int j = 0; j < kTransTileRowBlocks; ++j)
                        if (j == k) { cw[2 * j] = c_lo; cw[2 * j + 1] = c_hi; }
                    sbytes |= sbyte << (8 * k);
                } else {
                    scales_t[g] = (uint8_t)sbyte;
                    codes_t[g] = make_uint2(c_lo, c_hi);
                }
            }
            if (vec && (!EMUL || store_codes)) {
                const int64_t g0 = (c0 + c) * rblocks + rb0;
                store32B<true>(codes_t + g0, reinterpret_cast<const uint32_t(&)[8]>(cw));
                *reinterpret_cast<uint32_t*>(scales_t + g0) = sbytes;
            }
        };
        if (ncols == kTransTileCols && nrb == kTransTileRowBlocks && vec_ok) encode_column(std::true_type{});
        else if (c < ncols) encode_column(std::false_type{});
        if constexpr (EMUL) {
            __syncthreads();                         // the whole tile now holds dequantized values
            uint16_t* dst = out + rb0 * 16 * cols + c0;
            const int chunks_per_row = ncols / 8;
            for (int ch = threadIdx.x; ch < 16 * nrb * chunks_per_row; ch += blockDim.x) {
                const int r = ch / chunks_per_row, q = ch - r * chunks_per_row;
                *reinterpret_cast<uint4*>(dst + (int64_t)r * cols + q * 8) =
                    *reinterpret_cast<const uint4*>(stage + r * kTransTileCols + q * 8);
            }
        }
        __syncthreads();                             // the stage may be overwritten by the next prefetch
        ty = ty_next;
        tx = tx_next;
    }
}

// The amax pass of the transposed path with the Hadamard option: the maximum of the transformed column groups, published like amax_kernel's.  Bound by
// memory: a thread reads 16 rows of four columns, 8 bytes at a time (256 contiguous bytes per warp and row), the butterflies run on
// pairs of columns (h = 1, 2, 4, 8, packed add and fused subtract, the arithmetic of hadamard16_pairs), and 1/4 is applied to the maximum alone.
// A transformed value that is not a number (a NaN in the input, or sums beyond the largest float) makes a NaN of the tensor scale and does not go unseen.
// us, as the tile walk of the quantize kernel and as this: 8192 x 14336 45.5 / 37.6 (6.25 TB/s), 8192 x 4096 17.6 / 13.5, 4096 x 4096 10.9 / 7.6, 2048 x 4096 7.5 / 4.9.
// Three blocks per SM and no more of them: four (64 registers) spill, 46.7 us; several waves 38.4 - 39.7.
constexpr int kAmaxColumnsBlocks = 3;
__global__ void __launch_bounds__(256, kAmaxColumnsBlocks)
amax_columns_kernel(const uint2* __restrict__ in, int64_t rblocks, int64_t chunks, uint32_t sign_mask, unsigned long long* __restrict__ slot, uint32_t gen) {
    pdl_launch_dependents();
    // item i: row block i / chunks, columns 4 (i % chunks) ..; a thread's items are i, i + stride, ...
    const int64_t items = rblocks * chunks, stride = (int64_t)gridDim.x * blockDim.x;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t step_y = stride / chunks, step_x = stride - step_y * chunks;
    int64_t y = i / chunks, x = i - y * chunks;
    {   // before the wait (see prefetch_l2): a line of 128 bytes of one of the 16 rows per thread, two lines per warp and row
        const int64_t first = i - (threadIdx.x & 31) + 16 * (threadIdx.x & 1);
        if (first < items) {
            const int64_t fy = first / chunks;
            prefetch_l2(in + (fy * 16 + (threadIdx.x >> 1 & 15)) * chunks + (first - fy * chunks));
        }
    }
    pdl_wait();
    const uint64_t NEG1 = pack2(-1.0f, -1.0f);
    float m0 = 0.0f, m1 = 0.0f;
    for (; i < items; i += stride) {
        const uint2* at = in + y * 16 * chunks + x;
        uint2 w[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) w[r] = __ldg(at + r * chunks);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            uint64_t P[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const uint32_t v = (half ? w[r].y : w[r].x) ^ ((sign_mask >> r & 1u) ? 0x80008000u : 0u);
                P[r] = pack2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u));
            }
#pragma unroll
            for (int h = 1; h < 16; h <<= 1) {
#pragma unroll
                for (int base = 0; base < 16; base += 2 * h) {
#pragma unroll
                    for (int j = base; j < base + h; ++j) {
                        const uint64_t p = P[j], q = P[j + h];
                        P[j] = add2(p, q);
                        P[j + h] = fma2(q, NEG1, p);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < 16; r += 2) {
                float a, b, c, d;
                unpack2(P[r], a, b);
                unpack2(P[r + 1], c, d);
                m0 = max3abs_nan(m0, a, b);
                m1 = max3abs_nan(m1, c, d);
            }
        }
        y += step_y;
        x += step_x;
        if (x >= chunks) { x -= chunks; ++y; }
    }
    uint32_t local = __float_as_uint(__fmul_rn(max3abs_nan(m0, m1, m1), 0.25f));
    __shared__ uint32_t warp_max[8];
    local = __reduce_max_sync(0xFFFFFFFFu, local);
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = local;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t m = 0u;
#pragma unroll
        for (int v = 0; v < 8; ++v) m = max(m, warp_max[v]);
        atomicMax(slot, ((unsigned long long)gen << 32) | m);
    }
}

}  // namespace absq
