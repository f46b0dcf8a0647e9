"""The sum-factorised FP32 3D step on either side of the rule that shares a tile's planes among five
CTAs (tiles of 32 x 8 x 4 vertices on 304 places at orders 1 and 2, 152 at 3 and 4): a few tiles, between
one and two waves of them (shared), nearly one wave, and over two (not shared); ragged, odd, periodic
and zero-gradient.  One step against the plain FP64 step: populations within 3e-5 of the largest
deviation, as the other 3D tests; and the moments of the next collision, which the parts' sums give, through
a second step."""
import numpy as np
import pytest

from oracle import sllbm3d as o3

from .test_gpu_3d import _fields

pytestmark = pytest.mark.gpu

CASES = {   # cells, order, periodic, cv, isothermal
    "p1_few": ((40, 17, 9), 1, True, 2.5, False), "p1_one_wave": ((64, 64, 64), 1, True, 2.5, False),
    "p1_between": ((68, 60, 66), 1, False, 2.5, False), "p1_over": ((100, 66, 70), 1, True, 1.5, False),
    "p2_few": ((18, 9, 5), 2, False, 1.5, True), "p2_between": ((33, 33, 33), 2, True, 2.5, False),
    "p2_over": ((48, 33, 35), 2, False, 2.5, False),
    "p3_few": ((13, 5, 4), 3, False, 2.5, False), "p3_between": ((22, 22, 11), 3, True, 1.5, False),
    "p3_over": ((22, 22, 17), 3, False, 2.5, False),
    "p4_few": ((9, 5, 3), 4, True, 2.5, False), "p4_one_wave": ((16, 16, 8), 4, True, 2.5, False),
    "p4_between": ((16, 16, 9), 4, False, 2.5, False), "p4_over": ((24, 16, 14), 4, True, 2.5, False),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_against_the_plain_step(gpu_lib, name):
    import torch
    from paper_1910_13918_gb300.sllbm import BC_PERIODIC, BC_ZERO_GRADIENT, SLLBM3D
    cells, p, periodic, cv, iso = CASES[name]
    h = 1.0 / (cells[0] * p)
    box = tuple((0.0, c * p * h) for c in cells)
    runs = {}
    for prec in ("f64", "f32"):
        s = SLLBM3D(cells=cells, order=p, box=box, bc=(BC_PERIODIC if periodic else BC_ZERO_GRADIENT,) * 3,
                    dt=0.5 * h / 2.857 / 3 ** 0.5, tau=0.8, cv=cv, isothermal=iso, prec=prec)
        s.precompute()
        X, Y, Z = (t.cpu().numpy() for t in s.coords())
        f = list(_fields(X, Y, Z, box, 3))
        if iso:
            f[4] = np.ones_like(f[4])
        s.init(*f)
        s.step(1)
        st = s.get_state()
        s.step(1)
        runs[prec] = (st, s.get_state())
        assert s.kernel_name == ("stream3d" if prec == "f32" else "plain_f64")
        npop = s.npop
    w = torch.tensor(o3.d3q125()[1], device="cuda")[:, None, None, None]
    for a, b in zip(runs["f32"], runs["f64"]):
        for pop in range(npop):
            scale = float((b[pop] - (w if pop == 0 else (2 * cv - 3) * w)).abs().max())
            assert float((a[pop] - b[pop]).abs().max()) <= 3e-5 * scale, pop
