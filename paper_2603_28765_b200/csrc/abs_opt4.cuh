// Group-quantize kernel for the 4-bit formats (IF4, NVFP4) with the training options of Sec. 4.1:
// the 16-point random Hadamard transform and / or stochastic rounding (App. B).  Same arithmetic as the
// generic kernel, bit for bit, in the packed style of the round-to-nearest fast path: f32x2 butterflies
// for the transform stages that pair whole registers, f32x2 index-domain rounding, integer Horner packing.
#pragma once
#include "abs_fast4.cuh"

namespace absq {

constexpr float kMagic = 12582912.0f;                 // 1.5 * 2^23: x + kMagic leaves RNE(x) in the low mantissa bits
constexpr uint32_t kMagicBits = 0x4B400000u;

__device__ __forceinline__ uint64_t add2_rp(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rp.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2_rm(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2_rp(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rp.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// Eight magnitudes 0..7 (nibbles of m), negated in two's complement where bit 3 of the nibble of s is set (s has no other bits):
// 8 - m borrows from no neighbour, and its bit 3 flipped is 16 - m, or 0 for m = 0.
__device__ __forceinline__ uint32_t negate_nibbles(uint32_t m, uint32_t s) {
    const uint32_t neg = m & (s - (s >> 3));                 // the magnitudes to negate
    return (m ^ neg) | ((s - neg) ^ s);
}

// c + (-w) * (one 16-bit field of rnd): the field is picked, weighted and subtracted by one instruction.
template <int W, bool UPPER>
__device__ __forceinline__ uint32_t minus_field(uint32_t rnd, uint32_t c) {
    constexpr uint32_t weight = (uint32_t)(256 - W) << (UPPER ? 8 : 0);      // signed byte -W for the wanted field, 0 for the other
    uint32_t d;
    asm("dp2a.lo.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(rnd), "r"(weight), "r"(c));
    return d;
}

// Per-element work of one group under stochastic rounding (steps 3-10 of Fig. 3a with both candidates
// rounded stochastically, App. B).  rnd[i] holds the two 16-bit random fields h of elements 2i (low half)
// and 2i+1; u = (h + 1/2) * 2^-16.
//
// The rule "lo if a == lo, else hi iff u < (a - lo) / (hi - lo)" is a ceiling: with phi the grid's fractional-index
// map (grid point g_i -> i, linear in between), the rounded index is ceil(phi(a) - u).  Both candidates are formed on
// magnitudes -- an error and its square do not see a common sign of x, value and code -- and take u off as an integer:
//   E2M1: phi is linear in the bit pattern of a float with one mantissa bit and the smallest normal exponent at 1, so b =
//   bits(a * 2^-126) (rounded up; below 1 an FP32 subnormal) is phi(a) * 2^22, and the index is bits 22.. of
//   b + 2^22 - 33 - 64 h (2^22 u = 64 h + 32).  Those bits alone are the pattern of value * 2^-126.
//   Integer: the pattern of |z| + 65 - 2^-16 (rounded up; ulp 2^-17), minus 2 h, is that of 64 + k + a fraction, z = y * 7/6
//   rounded to FP32 as in the round-to-nearest path; an add that rounds down drops the fraction.
// Rounding up to a grid on which 2^22 u, or 2^17 u, lies crosses neither u nor an integer that the exact value does not reach.
// What bounds the kernels that call this is the arithmetic pipes, so the count of instructions: 36 -> 25 per pair of elements against three
// float pieces for phi, a float subtraction of u and signs put back on both values.  IF4, 8192 x 8192, 17/16 option, us before and after:
// rows with Hadamard 92.3 / 76.0, rows 84.0 / 69.9, columns with Hadamard 104.6 / 86.2; NVFP4 63.5 / 53.4, 53.4 / 47.1, 73.9 / 64.4.
// CLAMP: |y| may exceed 6 (then |z| 7; fl(6 * fp32(7/6)) is 7, so one clamp serves both).  It stays below 6 (1 + 7 * 2^-24), and neither index passes 7, with
// the 17/16 option, a scale byte that is neither subnormal nor saturated, and an alpha between 2^-120 and 2^117, which keeps 6 alpha, d and their
// reciprocals normal (alphas of supported tensors lie between 2^-112 and 2^117; a given alpha can be anything).  The clamp makes 6 of a y that is not a
// number, too; without it, such a y leaves its nibble.
__device__ __forceinline__ bool alpha_keeps_y_below_the_clamp(float alpha) {
    constexpr uint32_t kLow = (127u - 120u) << 23, kHigh = (127u + 117u) << 23;        // 2^-120, 2^117
    return __float_as_uint(alpha) - kLow <= kHigh - kLow;
}
template <bool HAS_INT, bool CLAMP>
__device__ __forceinline__ void encode_body4_sr(const float (&x)[16], const uint32_t (&rnd)[8], uint32_t sb, float d,
                                                float r, uint32_t& sbyte, uint32_t& c_lo, uint32_t& c_hi) {
    const uint64_t R2 = pack2(r, r);
    constexpr float kTiny = 1.17549435e-38f, kHuge = 8.507059173e37f;          // 2^-126, 2^126
    const uint64_t TINY = pack2(kTiny, kTiny), HUGE2 = pack2(kHuge, kHuge);
    const float c_pre = __uint_as_float(0x3F955555u);    // fp32(7/6)
    const float c_post = __uint_as_float(0x3F5B6DB7u);   // fp32(6/7)
    const float d_int = __fmul_rn(d, c_post);
    const uint64_t ND2 = pack2(-d, -d), NDI2 = pack2(-d_int, -d_int), CP2 = pack2(c_pre, c_pre);
    constexpr float kBase = 65.0f - 1.0f / 65536.0f;
    const uint64_t BASE = pack2(kBase, kBase), FLOOR = pack2(kMagic - 64.0f, kMagic - 64.0f), NMG = pack2(-kMagic, -kMagic);

    uint64_t accF[2], accI[2];
    uint32_t word[2], sign[2], kb[16];
#pragma unroll
    for (int hgrp = 0; hgrp < 2; ++hgrp) {
        float vs[8], xs[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = 8 * hgrp + 2 * i;
            xs[2 * i] = x[e]; xs[2 * i + 1] = x[e + 1];
            const uint32_t rw = rnd[e >> 1];
            const uint64_t X = pack2(fabsf(x[e]), fabsf(x[e + 1]));
            uint64_t Y = mul2(X, R2);                                          // E1 (step 3)
            if constexpr (CLAMP) {
                float y0, y1;
                unpack2(Y, y0, y1);
                Y = pack2(fminf(y0, 6.0f), fminf(y1, 6.0f));
            }
            // E2 under stochastic rounding
            float b0, b1, v0, v1;
            unpack2(mul2_rp(Y, TINY), b0, b1);
            constexpr uint32_t kOffset = (1u << 22) - 33u, kIndex = 0xFFC00000u;
            v0 = __uint_as_float(minus_field<64, false>(rw, __float_as_uint(b0) + kOffset) & kIndex);
            v1 = __uint_as_float(minus_field<64, true>(rw, __float_as_uint(b1) + kOffset) & kIndex);
            const uint64_t V = mul2(pack2(v0, v1), HUGE2);                     // value of the index (exact)
            unpack2(V, vs[2 * i], vs[2 * i + 1]);
            if constexpr (HAS_INT) {
                const uint64_t E = fma2(V, ND2, X);                            // E3 (steps 5-6), negated; squared below
                accF[hgrp] = (i == 0) ? mul2(E, E) : fma2(E, E, accF[hgrp]);
                // E4 (step 7) under stochastic rounding
                float z0, z1, k0, k1;
                unpack2(add2_rp(mul2(Y, CP2), BASE), z0, z1);
                z0 = __uint_as_float(minus_field<2, false>(rw, __float_as_uint(z0)));
                z1 = __uint_as_float(minus_field<2, true>(rw, __float_as_uint(z1)));
                const uint64_t KM = add2_rm(pack2(z0, z1), FLOOR);             // kMagic + k
                const uint64_t FI = fma2(add2(KM, NMG), NDI2, X);              // E5 (steps 8-9)
                accI[hgrp] = (i == 0) ? mul2(FI, FI) : fma2(FI, FI, accI[hgrp]);
                unpack2(KM, k0, k1);
                kb[e] = __float_as_uint(k0);
                kb[e + 1] = __float_as_uint(k1);
            }
        }
        word[hgrp] = e2m1x8_encode(vs);                                        // exact: the values are on the grid
        sign[hgrp] = e2m1x8_encode(xs) & 0x88888888u;                          // the sign bits alone
    }
    c_lo = word[0] | sign[0];
    c_hi = word[1] | sign[1];
    sbyte = sb;
    if constexpr (HAS_INT) {
        float f0, f1, f2, f3, i0, i1, i2, i3;
        unpack2(accF[0], f0, f1); unpack2(accF[1], f2, f3);
        unpack2(accI[0], i0, i1); unpack2(accI[1], i2, i3);
        const float E_fp = __fadd_rn(__fadd_rn(f0, f1), __fadd_rn(f2, f3));     // S1-S2 (step 10)
        const float E_int = __fadd_rn(__fadd_rn(i0, i1), __fadd_rn(i2, i3));
        const bool flag = E_int < E_fp;
        // magnitudes 0..7 by Horner on the raw sums (each holds kMagicBits + k), then two's complement where the sign is set
        constexpr uint32_t kConst = kMagicBits * 0x11111111u;
        uint32_t il = kb[7], ih = kb[15];
#pragma unroll
        for (int j = 6; j >= 0; --j) {
            il = il * 16u + kb[j];
            ih = ih * 16u + kb[8 + j];
        }
        il = negate_nibbles(il - kConst, sign[0]);
        ih = negate_nibbles(ih - kConst, sign[1]);
        c_lo = flag ? il : c_lo;
        c_hi = flag ? ih : c_hi;
        sbyte = sb | (flag ? 0x80u : 0u);
    }
}

// Threads of a block, and resident blocks per SM the kernel is compiled for (opt_grid says what it is launched for).  IF4 with stochastic rounding takes 91 to 94 registers: five blocks
// of 128 threads (20 warps) instead of two of 256 (8192 x 8192, us: 69.8 -> 66.1, with Hadamard 76.0 -> 73.9, emulation 82.1 -> 78.0; NVFP4 46.8 / 47.2, so it
// stays); the Hadamard-only kernels run best with three blocks of 256, the plain round-to-nearest one (used by the emulation pass only) with four.  A grid
// of one block per SM (kOnePass) has blocks of 256.
constexpr int opt_threads(bool has_int, bool sr, int src) { return has_int && sr && src != kOnePass ? 128 : 256; }
constexpr int opt_blocks_per_sm(bool has_int, bool sr, bool rht, int src) { return sr ? (opt_threads(has_int, sr, src) == 128 ? 5 : 2) : (rht ? 3 : 4); }

// Persistent grid-stride kernel, one group of 16 per thread and iteration, next group's 32 bytes fetched
// before the current one is encoded.  scale_mul is 17/16 with that option and 1 otherwise (times 1 is exact).
// EMUL = true is the emulation pass of Sec. 4.1 (every format was emulated by dequantizing right after
// quantizing): the group is decoded from the registers that hold its codes and scale, with the arithmetic of
// the dequantize kernel, and written to `out` as bf16; codes and scale bytes are stored only when
// `store_codes` is set.
template <bool HAS_INT, bool RHT, bool SR, int SRC, bool EMUL>
__global__ void __launch_bounds__(opt_threads(HAS_INT, SR, SRC), opt_blocks_per_sm(HAS_INT, SR, RHT, SRC))
quantize4_opt_kernel(const uint4* __restrict__ in, uint2* __restrict__ codes, uint8_t* __restrict__ scales,
                     const AlphaSrc alpha_src, int32_t ngroups, float scale_mul, uint32_t sign_mask,
                     const PhiloxKeys keys, uint64_t ctr_base, bool aligned32, uint4* __restrict__ out, bool out_aligned32,
                     bool store_codes) {
    pdl_launch_dependents();
    const int32_t stride = (int32_t)(gridDim.x * blockDim.x);
    int32_t g = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
    if (g < ngroups) prefetch_l2(in + 2 * (size_t)g);                  // before the wait: see prefetch_l2
    pdl_wait();
    uint32_t w[8], wn[8];
    const bool active = g < ngroups;
    if (active) {
        if (aligned32) load32B<true>(in + 2 * (size_t)g, w);
        else load32B<false>(in + 2 * (size_t)g, w);
    }
    uint32_t smask[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
        smask[i] = (((sign_mask >> (2 * i)) & 1u) << 15) | (((sign_mask >> (2 * i + 1)) & 1u) << 31);
    float alpha;                                                             // T2
    if constexpr (SRC == kOnePass && RHT) {
        auto bits = [&](const uint32_t (&r)[8]) {
            float x[16], m = 0.0f;
            hadamard16_packed(r, smask, x);
#pragma unroll
            for (int i = 0; i < 16; i += 2) m = max3abs(m, x[i], x[i + 1]);
            return __float_as_uint(m);
        };
        alpha = one_pass_alpha(alpha_src, thread_max_bits(w, in, g, stride, ngroups, aligned32, bits));
    } else {
        alpha = alpha_of<SRC>(alpha_src, w, in, g, stride, ngroups, aligned32);
    }
    __shared__ float2 scale_table[128];
    fill_scale_table(scale_table, alpha);                                    // G5 for every scale byte, once per block
    if (!active) return;
    const float inv_a6 = __frcp_rn(__fmul_rn(alpha, 6.0f));                  // T3
    // Scale bytes 8 .. 125 go without the clamp where the rest of encode_body4_sr's conditions hold.  (A number and not a truth value: kept over the loop, that took two
    // registers more, and the emulation pass of NVFP4 with Hadamard 7.6 us instead of 6.1, back to back at 1000 x 4096.)
    const uint32_t unclamped = scale_mul > 1.0f && alpha_keeps_y_below_the_clamp(alpha) ? 118u : 0u;
    while (true) {
        const int32_t gn = g + stride;
        const bool more = gn < ngroups;
        if (more) {
            if (aligned32) load32B<true>(in + 2 * (size_t)gn, wn);
            else load32B<false>(in + 2 * (size_t)gn, wn);
        }
        float x[16];
        if constexpr (RHT) {
            hadamard16_packed(w, smask, x);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                x[2 * i] = __uint_as_float(w[i] << 16);
                x[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
            }
        }
        uint32_t rnd[8];
        if constexpr (SR) {
            // Philox blocks 2g and 2g+1 hold the sixteen 16-bit fields of elements 16g .. 16g+15; ctr_base (even)
            // is the block index of the call's first element in the whole tensor (sr_index_offset / 8)
            const uint64_t i8 = ctr_base + (uint64_t)(uint32_t)g * 2u;
            const uint4 p0 = philox4x32_10((uint32_t)i8, (uint32_t)(i8 >> 32), keys);
            const uint4 p1 = philox4x32_10((uint32_t)i8 + 1u, (uint32_t)(i8 >> 32), keys);
            rnd[0] = p0.x; rnd[1] = p0.y; rnd[2] = p0.z; rnd[3] = p0.w;
            rnd[4] = p1.x; rnd[5] = p1.y; rnd[6] = p1.z; rnd[7] = p1.w;
        }
        // G1: group maximum with three-input max.
        const auto group_max = [&](auto max3) {
            const float m0 = max3(x[0], x[1], x[2]), m1 = max3(x[3], x[4], x[5]);
            const float m2 = max3(x[6], x[7], x[8]), m3 = max3(x[9], x[10], x[11]);
            const float m4 = max3(x[12], x[13], x[14]);
            return max3(max3(m0, m1, m2), max3(m3, m4, x[15]), x[15]);
        };
        const auto drop_nan = [](float a, float b, float c) { return max3abs(a, b, c); };
        const auto keep_nan = [](float a, float b, float c) { return max3abs_nan(a, b, c); };
        // G2-G3 (Eq. 2), with the 17/16 option folded into scale_mul; G5: d = Delta * alpha and 1 / d.
        uint32_t sb;
        float d, r;
        const auto scale_of = [&](float gmax) {
            sb = e4m3_encode(__fmul_rn(__fmul_rn(gmax, inv_a6), scale_mul));
            const float2 dr = scale_table[sb];
            d = dr.x;
            r = dr.y;
        };
        // With a NaN among them t is one and its byte 0x7F, which leads off the path without the clamp: no instruction more on that path (8192 x 8192,
        // before and after, us, with Hadamard: IF4 73.4 / 73.4, without 17/16 74.9 / 75.8, NVFP4 52.9 / 53.2); a test of its own there cost 2 - 3 %.
        if constexpr (SR) scale_of(group_max(keep_nan));
        else scale_of(group_max(drop_nan));
        uint32_t sbyte = 0u, c_lo = 0u, c_hi = 0u;
        if constexpr (SR) {
            // without the clamp where it cannot act (IF4 with Hadamard, 8192 x 8192: 77.9 -> 76.0 us; the transposed kernel, which
            // unrolls four groups, gained nothing from a second copy)
            if ((sb - 8u) < unclamped) {
                encode_body4_sr<HAS_INT, false>(x, rnd, sb, d, r, sbyte, c_lo, c_hi);
            } else {
                if (sb == 0x7Fu) scale_of(group_max(drop_nan));            // the scale is that of the numbers of the group
                if (sb != 0u) encode_body4_sr<HAS_INT, true>(x, rnd, sb, d, r, sbyte, c_lo, c_hi);      // G4: zero scale -> zeros
            }
        } else {
            if ((sb - 8u) >= 118u) {
                if (sb != 0u) encode_body4<HAS_INT, HAS_INT>(x, sb, d, r, sbyte, c_lo, c_hi);
            } else {
                encode_body4<HAS_INT, false>(x, sb, d, r, sbyte, c_lo, c_hi);
            }
        }
        if (!EMUL || store_codes) {
            scales[g] = (uint8_t)sbyte;
            codes[g] = make_uint2(c_lo, c_hi);
        }
        if constexpr (EMUL) {
            const bool is_int = HAS_INT && (sbyte & 0x80u);
            const float dd = is_int ? __fmul_rn(d, __uint_as_float(0x3F5B6DB7u)) : d;        // d * fp32(6/7) for integer groups
            const float addend = is_int ? -1032.0f : -0.0f;
            const uint64_t D2 = pack2(dd, dd);
            uint32_t lo[4], hi[4];
            dequant_word4<HAS_INT>(c_lo, is_int, addend, D2, lo);
            dequant_word4<HAS_INT>(c_hi, is_int, addend, D2, hi);
            const uint32_t o[8] = {lo[0], lo[1], lo[2], lo[3], hi[0], hi[1], hi[2], hi[3]};
            if (out_aligned32) store32B<true>(out + 2 * (size_t)g, o);
            else store32B<false>(out + 2 * (size_t)g, o);
        }
        if (!more) break;
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = wn[i];
        g = gn;
    }
}

}  // namespace absq
