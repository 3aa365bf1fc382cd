"""The head/tail split of the tensor-core products: both parts are TF32 values,
and together they are the operand to one unit of FP32."""

import numpy as np

from .native import build_native, run_native

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include "mma_tf32.cuh"
using namespace ams;
int main() {
    long loose = 0, off = 0, nan_lost = 0;
    uint32_t seed = 12345;
    for (long i = 0; i < 20000000; ++i) {
        seed = seed * 1664525u + 1013904223u;
        const uint32_t mant = i < (1 << 23) ? (uint32_t)i : seed >> 9;            // every mantissa, then random values
        const uint32_t e = i < (1 << 23) ? 127u : 30u + (seed >> 3) % 200u;
        const float x = f32_of_bits((seed & 0x80000000u) | e << 23 | mant);
        uint32_t hi, lo;
        split_tf32(x, hi, lo);
        loose += (hi & 0x1fffu) != 0 || (lo & 0x1fffu) != 0;
        const double unit = std::ldexp(1.0, (int)e - 127 - 23);
        off += !(std::fabs((double)x - (double)f32_of_bits(hi) - (double)f32_of_bits(lo)) <= unit);
    }
    const uint32_t special[] = {0x7f800000u, 0xff800000u, 0x7fc00000u, 0x7fffffffu, 0xffffffffu, 0x7f800001u};
    for (uint32_t b : special) {
        uint32_t hi, lo;
        split_tf32(f32_of_bits(b), hi, lo);
        nan_lost += !std::isnan(f32_of_bits(lo));
    }
    uint32_t hi, lo;
    split_tf32(0.f, hi, lo);
    std::printf("%ld %ld %ld %d\n", loose, off, nan_lost, hi == 0 && lo == 0);
}
"""


def test_parts_are_tf32_and_sum_to_the_operand(tmp_path):
    assert run_native(build_native(tmp_path, SOURCE)) == ["0 0 0 1"]


def test_products_of_split_operands():
    """tail*head + head*tail + head*head is a*b to 2^-21: the dropped tail*tail and the operands' last units."""
    rng = np.random.default_rng(3)
    a, b = (rng.standard_normal(200000).astype(np.float32) for _ in range(2))

    def split(x):
        h = ((x.view(np.uint32) + np.uint32(0x1000)) & np.uint32(0xffffe000)).view(np.float32)
        t = ((x - h).view(np.uint32) & np.uint32(0xffffe000)).view(np.float32)
        return h.astype(np.float64), t.astype(np.float64)
    (ah, at), (bh, bt) = split(a), split(b)
    exact = a.astype(np.float64) * b.astype(np.float64)
    assert (np.abs(at * bh + ah * bt + ah * bh - exact) <= 2.0 ** -21 * np.abs(exact)).all()
