// Building blocks of the tensor-core products (abs_gemm.cu, abs_skinny.cuh): mbarriers, TMA loads, tensor memory, the
// block-scaled FP4 MMA, and the split of integer codes into two E2M1 values.
#pragma once
#include "abs_device.cuh"

#include <cuda.h>

namespace absq {

constexpr int kTileM = 128, kTileN = 128;
constexpr int kStageK = 256;                       // elements of K of one TMA box: 128 bytes of packed codes per row
constexpr int kMmaK = 64;                          // K of one tcgen05.mma kind::mxf4nvf4
constexpr int kPlaneBytes = kTileM * kStageK / 2;  // 16 KiB: one box (128 rows x 128 bytes) of one plane of one operand
// IF4: the accumulator H H of a tile is summed in the tensor core over at most kChunkK of K, and the epilogue adds the chunks in
// registers; H L + L H and L L, which count a seventh and less, run over the whole of K.  A long chain rounds more with every
// step where scales span a wide range, while adding chunks of H H, whose values lie on a coarse grid, mostly does not round and
// adding all three chunk by chunk does.  2-norm against 64 bits, K = 14336, activations x weights / gradients with Hadamard
// and stochastic rounding: 3.8e-8 / 2.0e-7; all three chunk by chunk 5.6e-8 / 2.2e-7; the nine-MMA split, one chain, 4.2e-8 / 1.0e-6.
// (Both operands of one sign: 1.2e-7, 6.1e-8 and 4.1e-7.)  A hand-over of H H costs less than the end of a tile, once per 4096 of K.
constexpr int kChunkK = 4096;
constexpr uint64_t kWaitLimitNs = 1000000000ull;   // one second: how long an mbarrier wait polls before the block gives up

// Splits eight integer codes (two's complement nibbles of one word) into the planes H and L (see abs_gemm.cu).  With sign
// s and magnitude m = |k| of each nibble, m = 0 .. 8: one byte permute looks up four magnitudes in a table of bytes
// h | l' << 4, where h is the E2M1 code of 0, 1, 2, 3, 4, 4, 6, 6 and l' that of 0, 1, 2, 3, 4, 2, 6, 0 with bit 3 set where l
// has the sign of k (5: 4 + 2/7) and not where it has the other (1 - 1/7, ...).  m = 8 (the most negative code, which no
// quantizer writes but dequantize reads as -8) selects, by the permute's sign mode, the sign of byte 0: 0xFF, which is
// h = -6, l = -6 once the signs are in.
__device__ __forceinline__ void split_int_word(uint32_t w, uint32_t& h, uint32_t& l) {
    constexpr uint32_t kLo = 0x55442280u, kHi = 0x0777C666u;
    const uint32_t s = w & 0x88888888u, neg = s >> 3;
    const uint32_t m = (w ^ (neg * 15u)) + neg;                      // |k| per nibble: no carry from one into the next
    uint32_t b0, b1;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(b0) : "r"(kLo), "r"(kHi), "r"(m));
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(b1) : "r"(kLo), "r"(kHi), "r"(m >> 16));
    // even bytes: h (l') of two neighbours in the two nibbles; odd bytes are not used
    const uint32_t x0 = b0 >> 4, x1 = b1 >> 4;
    const uint32_t h0 = (b0 & 0x0F0F0F0Fu) | (x0 & 0xF0F0F0F0u), h1 = (b1 & 0x0F0F0F0Fu) | (x1 & 0xF0F0F0F0u);
    const uint32_t l0 = (x0 & 0x0F0F0F0Fu) | ((b0 >> 8) & 0xF0F0F0F0u), l1 = (x1 & 0x0F0F0F0Fu) | ((b1 >> 8) & 0xF0F0F0F0u);
    h = __byte_perm(h0, h1, 0x6420) | s;
    l = __byte_perm(l0, l1, 0x6420) ^ s ^ 0x88888888u;
}

// ----------------------------------------------------------------------------- PTX building blocks

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}
__device__ __forceinline__ uint64_t global_timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// One lane of the (converged) warp, the same at every call.
__device__ __forceinline__ bool elect_one() {
    uint32_t one;
    asm volatile("{ .reg .pred p; elect.sync _|p, 0xFFFFFFFF; selp.u32 %0, 1, 0, p; }" : "=r"(one));
    return one != 0;
}
// Wait for the phase with the given parity, bounded in time (a try_wait may itself sleep for a while, so counting
// polls would not bound it); false when the limit ran out.  Reading the timer between polls also keeps the waiting warps from
// crowding the others: with 64 polls before the first read a 1000 x 14336 x 4096 NVFP4 product took 6 % longer.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_timer_ns();
    do {
        if (mbar_try_wait(bar, parity)) return true;
    } while (global_timer_ns() - t0 < kWaitLimitNs);
    return false;
}
// The same by all lanes of a warp, with one answer.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity) { return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity)); }
// One 2-D tile (inner coordinate x in bytes, outer coordinate y in rows) from a tensor map into shared memory.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int32_t x, int32_t y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}
// `bytes` contiguous bytes (a multiple of 16, both addresses 16-byte aligned) into shared memory.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// Requests such a tile into the L2.
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int32_t x, int32_t y) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" :: "l"(map), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t smem_result, uint32_t columns) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_result), "r"(columns) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() { asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_free(uint32_t addr, uint32_t columns) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(addr), "r"(columns) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Arrives on the mbarrier once every tcgen05 operation this thread issued before has completed.
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(bar) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T, 128 x 128 x 64, E2M1 operands, one UE4M3 scale per 16 elements read from tensor memory.
// What happens to the A operand in the tensor core's collector buffer: read from shared memory and dropped, read and
// kept (kFill), taken from the buffer and dropped (kLastUse).  An MMA that takes A from the buffer reads only B from shared
// memory.
enum Collector { kDiscard, kFill, kLastUse };
template <Collector C = kDiscard>
__device__ __forceinline__ void tc_mma_nvf4(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, bool accumulate,
                                            uint32_t sfa_tmem, uint32_t sfb_tmem) {
#define ABS_MMA_NVF4(USAGE)                                                                                              \
    asm volatile("{ .reg .pred p; setp.ne.b32 p, %4, 0;\n"                                                               \
                 "  tcgen05.mma.cta_group::1.kind::mxf4nvf4.block_scale.block16" USAGE " [%0], %1, %2, %3, [%5], [%6], p; }" \
                 :: "r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"((uint32_t)accumulate), "r"(sfa_tmem), "r"(sfb_tmem) \
                 : "memory")
    if constexpr (C == kFill) ABS_MMA_NVF4(".collector::a::fill");
    else if constexpr (C == kLastUse) ABS_MMA_NVF4(".collector::a::lastuse");
    else ABS_MMA_NVF4("");
#undef ABS_MMA_NVF4
}
// 32 lanes x 32 columns of 32 bits: thread t of the warp gets columns c .. c+31 of lane (warp % 4) * 32 + t.
__device__ __forceinline__ void tmem_load32(uint32_t addr, uint32_t (&r)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(addr) : "memory");
}
// The same with 16 columns.
__device__ __forceinline__ void tmem_load16(uint32_t addr, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(addr) : "memory");
}
// The same with 8 columns.
__device__ __forceinline__ void tmem_load8(uint32_t addr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr) : "memory");
}
// Two FP32 values rounded to nearest even bf16, the first in the low half.
__device__ __forceinline__ uint32_t bf16x2_bits(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// Sixteen neighbouring columns of a row of C times `scale`, from column index `at` on: 64 (FP32) or 32 (bf16) contiguous bytes of one thread, which takes a run
// of such columns in order, first to last.  Whole sectors leave at a time: where C is 32-byte aligned as they are, otherwise (C is 16-byte aligned, rows
// are whole sectors long) the second half of 32 bytes is held back for the first of the next, and only the ends of the run are half sectors.  (As
// two 16-byte stores each, whose sectors the next one completes, FP32 products into such a C took up to 1.4 times as long: NVFP4 4096 x 4096 x 512 20.2 us by lines
// turned through shared memory, 28.5 so, 18.3 held back; 2048 x 4096 x 4096 bf16 27.3, 26.2, 24.0.)
// WHOLE: whether C is 32-byte aligned.  Where the choice lies follows from what it costs aligned outputs.  IF4, FP32: per 16 columns nothing (0.8 % at
// 4096 x 4096 x 512), around all 64 of a thread 0.5 - 1 %, by selects instead of a branch 0.1 - 0.8 %, per 32 bytes 2.5 % at 4096 x 4096 x 512.  NVFP4: per 32 columns, and in the
// pairs of tiles per tile, nothing; by selects 2 % in bf16 at 1000 x 4096 x 1024.
// keep_max: the larger of out_max and the bf16 magnitudes written, per half word.
template <bool OUT_BF16, bool WHOLE>
__device__ __forceinline__ void store_columns16(void* c_out, size_t at, const float* v, float scale, bool first, bool last, uint4& held, bool keep_max,
                                                uint32_t& out_max) {
    constexpr int kPieces = OUT_BF16 ? 1 : 2;
#pragma unroll
    for (int q = 0; q < kPieces; ++q) {
        uint32_t o[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if constexpr (OUT_BF16) {
                o[e] = bf16x2_bits(__fmul_rn(v[2 * e], scale), __fmul_rn(v[2 * e + 1], scale));
                if (keep_max) out_max = __vmaxu2(out_max, o[e] & 0x7FFF7FFFu);
            } else {
                o[e] = __float_as_uint(__fmul_rn(v[8 * q + e], scale));
            }
        }
        uint8_t* const to = reinterpret_cast<uint8_t*>(c_out) + at * (OUT_BF16 ? 2 : 4) + 32 * q;
        if constexpr (WHOLE) {
            store32B<true>(to, o);
        } else {
            if (first && q == 0) {
                *reinterpret_cast<uint4*>(to) = make_uint4(o[0], o[1], o[2], o[3]);
            } else {
                const uint32_t sector[8] = {held.x, held.y, held.z, held.w, o[0], o[1], o[2], o[3]};
                store32B<true>(to - 16, sector);
            }
            held = make_uint4(o[4], o[5], o[6], o[7]);
            if (last && q == kPieces - 1) *reinterpret_cast<uint4*>(to + 16) = held;
        }
    }
}
__device__ __forceinline__ void tmem_load_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// 32 lanes x 16 columns of 32 bits: thread t of the warp writes columns c .. c+15 of lane (warp % 4) * 32 + t.
__device__ __forceinline__ void tmem_store16(uint32_t addr, const uint4& a, const uint4& b, const uint4& c, const uint4& d) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 :: "r"(addr), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w), "r"(c.x), "r"(c.y),
                    "r"(c.z), "r"(c.w), "r"(d.x), "r"(d.y), "r"(d.z), "r"(d.w)
                 : "memory");
}
__device__ __forceinline__ void tmem_store_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Magnitudes of sixteen scale bytes: an integer group carries its flag in the sign bit.
__device__ __forceinline__ uint4 mask_scales(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    constexpr uint32_t kMag = 0x7F7F7F7Fu;
    return make_uint4(a & kMag, b & kMag, c & kMag, d & kMag);
}

// Shared-memory matrix descriptors (64 bits): start address, leading / stride byte offsets (all in 16-byte units),
// descriptor version 1 (Blackwell) in bits 46-47, swizzle mode in bits 61-63.
//   operand tiles: K-major rows of 128 bytes, 128-byte swizzle (mode 2), 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t operand_desc(uint32_t smem_addr) {
    return (uint64_t)((smem_addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
           ((uint64_t)2 << 61);
}
// Instruction descriptor of kind::mxf4nvf4: A and B E2M1 (format 1, bits 7-9 and 10-12), both K-major, N / 8 in bits
// 17-22, scale format UE4M3 (bit 23 = 0), M / 16 in bits 24-28, dense, K = 64 (bit 31 = 0), scale ids 0.
constexpr uint32_t kInstrDesc = (1u << 7) | (1u << 10) | ((uint32_t)(kTileN >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);

}  // namespace absq
