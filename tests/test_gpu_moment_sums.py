"""The mass and energy sums of FP32 and BF16 states keep FP64 precision for any populations: random
deviations spread over ten decades, the same on every vertex, against exact rational sums.  The
bound is that of an FP64 evaluation: 32 roundings (5 to combine a row, column or g sum, at most 9 in
the weighted terms, 9 + 9 over the 9 vertices and their weights) of the sum of the terms' magnitudes.
And sums beyond the FP32 range stay finite, as FP64 sums of the same values are."""
import dataclasses
from fractions import Fraction as F

import numpy as np
import pytest

from oracle import sllbm as o
from paper_1910_13918_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _sim(prec, cv):
    from paper_1910_13918_gb300.sllbm import SLLBM
    s = SLLBM.from_workload(dataclasses.replace(W.tgv16(), order=1, cv=cv).resized(3, 3), prec=prec)
    s.precompute()
    return s


def _check(s, cv, pops):
    import torch
    st = torch.tensor(pops, dtype=torch.float64)[:, :, None, None].expand(-1, -1, s.ny, s.nx).to(s.state_dtype).cuda()
    s.set_state(st)
    m = s.moments()
    vals = st[:, :, 0, 0].double().cpu().numpy()
    A = sum(F(float(a)) for a in s.vertex_weights().cpu().numpy().reshape(-1))
    xi = o.d1q5()[0]
    f, g = vals[0], (vals[1] if s.npop == 2 else np.zeros(25))
    e = [F(float(xi[i // 5])) ** 2 + F(float(xi[i % 5])) ** 2 for i in range(25)]
    mass = [F(1)] + [F(float(v)) for v in f]
    energy = [F(2 * cv)] + [F(float(v)) * c for v, c in zip(f, e)] + [F(float(v)) for v in g]
    for got, terms in ((m["mass"], mass), (2 * F(m["energy"]), energy)):
        ref, scale = A * sum(terms), A * sum(abs(t) for t in terms)
        assert abs(F(got) - ref) <= F(32, 2 ** 53) * scale, float(abs(F(got) - ref) / scale)


@pytest.mark.parametrize("prec", ["f32", "bf16"])
@pytest.mark.parametrize("cv", [2.5, 1.0])
def test_sums_of_populations_over_ten_decades(gpu_lib, prec, cv):
    s = _sim(prec, cv)
    rng = np.random.default_rng(11)
    for _ in range(200):   # positive: density and temperature are too
        _check(s, cv, 10.0 ** rng.uniform(-10, 0, (s.npop, 25)))


def test_sums_of_g_over_eight_decades(gpu_lib):
    s = _sim("f32", 2.5)
    rng = np.random.default_rng(12)
    for _ in range(200):
        _check(s, 2.5, 10.0 ** rng.uniform((-10, -4), (0, 4), (25, 2)).T)


@pytest.mark.parametrize("prec", ["f32", "bf16"])
def test_sums_beyond_the_fp32_range(gpu_lib, prec):
    s = _sim(prec, 2.5)
    pops = np.full((2, 25), 1e-3)
    pops[:, [0, 5, 6, 12, 18]] = 2e38
    _check(s, 2.5, pops)
