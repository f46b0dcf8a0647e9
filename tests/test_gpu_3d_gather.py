"""The one-launch gather form of the FP32 3D step on grids of more than one wave of blocks (over
77,824 vertices), every order, with departures that leave the neighbouring cells, next to equilibrium:
deviations of 1e-4 of the lattice weights.  One step against the plain FP64 step from the same
fields: populations within 3e-5 of the largest deviation, as in the other 3D tests.  (Forming the
equilibrium through a sum with its leading 1 would leave 2^-24 of the weights, over ten times that.)"""
import numpy as np
import pytest

from oracle import sllbm as o
from oracle import sllbm3d as o3

pytestmark = pytest.mark.gpu

CASES = {"p1": (44, 1, 1.2), "p2": (22, 2, 0.7), "p3": (15, 3, 0.5), "p4": (11, 4, 0.5)}   # cells, order, reach in cells


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("cv", [2.5, 1.5])
def test_near_equilibrium_against_the_plain_step(gpu_lib, name, cv):
    from paper_1910_13918_gb300.sllbm import BC_PERIODIC, SLLBM3D
    n, p, reach = CASES[name]
    dt = reach / n / max(o.d1q5()[0])
    st = {}
    for prec in ("f32", "f64"):
        s = SLLBM3D(cells=(n, n, n), order=p, box=((0.0, 1.0),) * 3, bc=(BC_PERIODIC,) * 3, dt=dt, tau=0.8, cv=cv, prec=prec)
        s.precompute()
        X, Y, Z = (2 * np.pi * t.cpu().numpy() for t in s.coords())
        s.init(1 + 1e-4 * np.sin(X) * np.cos(Y), 1e-4 * np.sin(Y), 5e-5 * np.cos(Z), 4e-5 * np.sin(X), 1 + 1e-4 * np.cos(X + Z))
        s.step(1)
        st[prec] = s.get_state().cpu().numpy()
        assert s.kernel_name == ("gather_f32" if prec == "f32" else "plain_f64")
    _, w = o3.d3q125()
    for pop, lat in enumerate((w, (2 * cv - 3) * w)[: s.npop]):
        scale = np.max(np.abs(st["f64"][pop] - lat[:, None, None, None]))
        err = np.max(np.abs(st["f32"][pop] - st["f64"][pop]))
        assert err <= 3e-5 * scale, (pop, err / scale)
