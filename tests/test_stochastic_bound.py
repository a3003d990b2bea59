"""The bound that lets the 4-bit row kernels with stochastic rounding and the 17/16 factor leave the clamp of |y| out (csrc/abs_opt4.cuh), over the scale bytes and
tensor scales for which they do: the steps up to the two indices, in the FP32 roundings of the kernel, where the scale is rounded down the furthest."""
import os
import re

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_28765_b200", "csrc")
F = np.float32


def _alphas(rng, low, high, n):
    edges = [F(2.0) ** F(low), np.nextafter(F(2.0) ** F(low), F(np.inf)), F(2.0) ** F(high), np.nextafter(F(2.0) ** F(high), F(0))]
    return np.concatenate([np.array(edges, F), np.exp2(rng.uniform(low, high, n)).astype(F)])


def test_no_index_leaves_its_nibble_without_the_clamp():
    text = open(os.path.join(CSRC, "abs_opt4.cuh")).read()
    low, high = re.search(r"kLow = \(127u - (\d+)u\) << 23, kHigh = \(127u \+ (\d+)u\) << 23", text).groups()
    alphas = _alphas(np.random.default_rng(1), -int(low), int(high), 4000)
    with np.errstate(over="ignore", under="ignore"):
        inv_a6 = F(1.0) / (alphas * F(6.0))
        tiny = np.finfo(F).tiny
        assert bool(np.isfinite(inv_a6).all()) and float(inv_a6.min()) >= tiny
        worst = 0.0
        for byte in range(8, 126):
            e, m = byte >> 3, byte & 7
            scale = F((1 + m / 8) * 2.0 ** (e - 7))
            middle = float((1 + (m + 0.5) / 8) * 2.0 ** (e - 7))         # a target up to here may be rounded down to this byte
            d = scale * alphas
            r = F(1.0) / d
            assert float(d.min()) >= tiny and float(r.min()) >= tiny and bool(np.isfinite(r).all())
            # the largest FP32 maxima whose target, rounded twice, does not pass the middle (finer than bf16 maxima, as after the transform)
            g = (middle / 1.0625 / inv_a6.astype(np.float64)).astype(F)
            for _ in range(6):
                up = np.nextafter(g, F(np.inf))
                fits = ((up * inv_a6) * F(1.0625)).astype(np.float64) <= middle
                g = np.where(fits & np.isfinite(up), up, g)
            for _ in range(8):
                g = np.where(((g * inv_a6) * F(1.0625)).astype(np.float64) > middle, np.nextafter(g, F(0)), g)
            ok = np.isfinite(g)
            y = (g * r)[ok]
            worst = max(worst, float(y.max()))
            # E2M1: bits(y * 2^-126) = phi(y) * 2^22 for y in [4, 8); the index stays 7 where bits + 2^22 - 33 is below 8 * 2^22
            bits = np.maximum(y, F(4.0)).view(np.uint32).astype(np.int64) - (126 << 23)
            assert int(bits.max()) + (1 << 22) - 33 < 8 << 22
            # integer: |z| + 65 - 2^-16 rounded up to the grid of 2^-17; below 72 the magnitude is at most 7
            z = (y * np.uint32(0x3F955555).view(F)).astype(np.float64)
            assert float((np.ceil((z + 65 - 2.0 ** -16) * 2.0 ** 17) * 2.0 ** -17).max()) < 72
        assert 6.0 < worst <= 6.0 * (1 + 7 * 2.0 ** -24)
