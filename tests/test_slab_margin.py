"""The walks' box test, entry <= exit kSlabMargin from centres, half extents (FP16, rounded up) and reciprocals to
one ulp, passes over no more boxes whose edge a ray just meets than the test it stands for: lo and hi
planes, IEEE reciprocals and a margin of 5e-7.  Both are carried out here in FP32, FMAs in FP64 rounded
once, on boxes of a room's, a street's and a city's size."""
import os
import re

import numpy as np
import pytest

from paper_2208_10009_gb300 import build

f = np.float32


def _margin():
    src = open(os.path.join(build.CSRC, "sbr_device.cuh")).read()
    m = re.search(r"kSlabMargin = ([0-9.]+)f;", src)
    return f(m.group(1)) if m else f(re.search(r"tcull = tmax \* ([0-9.]+)f;", src).group(1))


def _fma(a, b, c):
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(f)


@pytest.mark.parametrize("size,lo_ext,hi_ext", [(10, 0.5, 5), (10, 5, 50), (300, 0.5, 5), (300, 5, 50), (300, 100, 1000),
                                                (3300, 0.5, 5), (3300, 5, 50), (3300, 100, 1000)])
@pytest.mark.parametrize("flat", [False, True])
def test_no_more_edges_missed(size, lo_ext, hi_ext, flat):
    rng, n = np.random.default_rng(int(size + hi_ext)), 600_000
    quarter = lambda x: (np.round(x * 4) / 4).astype(f)          # coordinates as a plan has them
    lo = quarter(rng.uniform(0, size, (n, 3)))
    hi = lo + quarter(np.exp(rng.uniform(np.log(lo_ext), np.log(hi_ext), (n, 3))) + 0.25)
    if flat:                                                     # a wall
        hi[:, 0] = lo[:, 0]
    p = lo + (hi - lo) * rng.random((n, 3))
    p[:, 0] = np.where(rng.random(n) < 0.5, lo[:, 0], hi[:, 0])  # on two planes of the box: its edge
    p[:, 1] = np.where(rng.random(n) < 0.5, lo[:, 1], hi[:, 1])
    d = rng.normal(size=(n, 3))
    d = (d / np.linalg.norm(d, axis=1)[:, None]).astype(f)
    o = (p - d.astype(np.float64) * 10 ** rng.uniform(0, 3, (n, 1))).astype(f)
    a, b = (lo.astype(np.float64) - o) / d, (hi.astype(np.float64) - o) / d
    met = np.minimum(a, b).max(1) <= np.maximum(a, b).min(1)
    inv = (f(1) / d).astype(f)
    a, b = _fma(lo, inv, -(o * inv)), _fma(hi, inv, -(o * inv))
    planes = np.minimum(a, b).max(1) <= np.maximum(a, b).min(1) * f(1.0000005)
    off = rng.integers(-1, 2, inv.shape)                         # an ulp either way
    inv = np.where(off == 0, inv, np.nextafter(inv, np.where(off > 0, f(np.inf), f(-np.inf)))).astype(f)
    c = (0.5 * (lo.astype(np.float64) + hi)).astype(f)
    need = np.maximum(hi - c.astype(np.float64), c.astype(np.float64) - lo)
    h = need.astype(np.float16)
    h = np.where(h.astype(np.float64) < need, np.nextafter(h, np.float16(np.inf)), h).astype(f)
    t = _fma(c, inv, -(o * inv))
    centres = _fma(h, -np.abs(inv), t).max(1) <= _fma(h, np.abs(inv), t).min(1) * _margin()
    assert met.sum() > n / 3
    assert np.sum(met & ~centres) <= np.sum(met & ~planes)
