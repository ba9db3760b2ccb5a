"""The device GELU's polynomial, evaluated on the host in FP32 as the kernel does.

The coefficients are read from the header; fused multiply-adds are formed in FP64 and
rounded once. Bound: half an ulp of a result below 8 (2^-22 = 2.4e-7), and on z t, at
most 0.17, the rounding of the exponent (|z P(|z|) - 1| < 8 where it counts, 2.4e-7 ln 2
times 0.1) and the 2^-22 of the hardware's power of two: 6e-8 together. From |z| = 8 on
the subtracted part is below 1e-14 and the result is max(z, 0) to half an ulp.
"""
import math
import pathlib
import re

import numpy as np
import pytest

HEADER = pathlib.Path(__file__).resolve().parents[1] / "paper_2201_10132_gb300" / "csrc" / "tfkt_mlp.cuh"


def _gelu(z):
    body = re.search(r"GELU_P\[10\] = \{(.*?)\}", HEADER.read_text(), re.S).group(1)
    c = np.array([float(v.rstrip("f")) for v in body.replace("\n", " ").split(",")]).astype(np.float32)
    assert c.size == 10
    fma = lambda a, b, d: (a.astype(np.float64) * b + np.float64(d)).astype(np.float32)
    a = np.abs(z)
    with np.errstate(over="ignore", invalid="ignore"):
        p = np.full_like(a, c[9])
        for k in range(8, -1, -1):
            p = fma(p, a, c[k])
        t = np.exp2(fma(p, a, -1.0).astype(np.float64)).astype(np.float32)
        return (-t.astype(np.float64) * np.minimum(a, np.float32(3e38)) + np.maximum(z, np.float32(0))).astype(np.float32)


@pytest.mark.parametrize("lo, hi", [(-8.0, -4.0), (-4.0, -0.5), (-0.5, 0.5), (0.5, 4.0), (4.0, 8.0)])
def test_gelu_against_fp64(lo, hi):
    z = np.linspace(lo, hi, 20001).astype(np.float32)
    exact = np.array([0.5 * v * math.erfc(-v / math.sqrt(2.0)) for v in z.astype(np.float64)])
    assert np.abs(_gelu(z) - exact).max() <= 2.0 ** -22 + 6e-8


def test_gelu_tails_and_specials():
    z = np.array([8.0, 13.0, 60.0, 1e4, 1e10, 3e38, np.inf], np.float32)
    assert np.array_equal(_gelu(z), z)
    assert np.abs(_gelu(-z)).max() < 1e-13
    assert _gelu(np.array([0.0], np.float32))[0] == 0.0
    assert np.isnan(_gelu(np.array([np.nan], np.float32)))[0]
