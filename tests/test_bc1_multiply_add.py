"""The division of a BC1 palette numerator by 3 (four colours) or 2 (three) as one FP32
multiply-add on 2^23 + numerator (csrc/common.cuh, bc1_texel_f), for every numerator:
the constants are read from the source, and the products and sums are exact in
double precision (48 and 50 bits), so one conversion gives the FMA's rounding."""
import os
import re

import numpy as np

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_06040_gb300", "csrc", "common.cuh")


def _fma(f, scale, add):
    return (f * np.float64(np.float32(scale)) + np.float64(np.float32(add))).astype(np.float32).astype(np.float64)


def test_palette_divisions_are_one_multiply_add():
    text = open(SRC).read()
    scale = re.search(r"b\.scale = four \? 1\.0f / 3\.0f : ([0-9.]+)f;", text).group(1)
    add4, add3 = re.search(r"b\.add = four \? ([0-9.]+)f : ([0-9.]+)f;", text).groups()
    base = float(re.search(r"kTexelBase = ([0-9.]+)f;", text).group(1))
    assert base == 2.0 ** 23 + 2.0 ** 22
    num = np.arange(1, 3 * 255 + 2)   # a0 e0 + a1 e1 + 1 with weights that add to 3
    assert np.array_equal(_fma(2.0 ** 23 + num, np.float32(1) / np.float32(3), float(add4)), base + num // 3)
    half = np.arange(0, 2 * 255 + 1)  # a0 e0 + a1 e1 with weights that add to 2, doubled, + 1
    assert np.array_equal(_fma(2.0 ** 23 + 2 * half + 1, float(scale), float(add3)), base + (half + 1) // 2)
