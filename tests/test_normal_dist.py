"""The block-tiled forward's normal distribution function (csrc/tile.cuh), in fp32 on the CPU, against the error that it states (with correctly rounded
exponential and division; the hardware's are not modelled)."""
import math
import pathlib
import re

import numpy as np

SOURCE = pathlib.Path(__file__).resolve().parent.parent / "paper_2608_21308_b200" / "csrc" / "tile.cuh"


def test_normal_distribution_function_is_within_its_stated_error():
    text = SOURCE.read_text()
    body = text[text.index("void normal_dist("):]
    body = body[:body.index("\n}\n")]
    coef = [np.float32(c) for c in re.findall(r"(-?\d\.\d{9})f", body)]  # from the highest degree down
    assert len(coef) == 10
    z = np.concatenate([np.linspace(-20, 20, 200001), np.geomspace(1e-30, 1, 1000), -np.geomspace(1e-30, 1, 1000)]).astype(np.float32)
    x = np.float32(0.70710678118) * np.abs(z)
    x2 = x * x

    def fma(a, b, c):
        return (a.astype(np.float64) * np.asarray(b, np.float64) + np.float64(c)).astype(np.float32)

    t = np.float32(1) / fma(x, 0.5, 1.0)
    p = np.full_like(t, coef[0])
    for c in coef[1:]:
        p = fma(t, p, c)
    q = np.float32(0.5) * t * np.exp(p - x2)
    cdf = np.where(z < 0, q, np.float32(1) - q).astype(np.float64)
    exact = np.array([0.5 * math.erfc(-float(v) / math.sqrt(2.0)) for v in z])
    assert np.max(np.abs(cdf - exact)) <= 2.6e-7
    # The tail keeps its relative accuracy: the arguments of the exponential, up to 87, are rounded to 2^-24 of their size three times (x,
    # whose error the square doubles, x^2, and the difference)
    tail = (z < 0) & (exact > 1e-37)
    assert np.max(np.abs(cdf[tail] / exact[tail] - 1)) <= 4 * 87 * 2.0 ** -24 + 1e-6
