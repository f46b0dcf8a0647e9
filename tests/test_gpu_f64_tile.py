"""The tile form of the plain FP64 step at the edges of its range: every order, ragged and tiny grids,
periodic, clamped and mixed axes, one population, the isothermal equilibrium, and time steps from
one whose departures stay in the cell to one whose window no longer fits (the gather form), against
the oracle's populations after 3 steps (1e-11 of the largest, as the other FP64 tests)."""
import dataclasses

import numpy as np
import pytest

from paper_1910_13918_gb300 import workloads as W

from . import helpers as H
from .test_gpu_parity import TOL_F64, gpu_run

pytestmark = pytest.mark.gpu

ZG, PER = W.ZERO_GRADIENT, W.PERIODIC


def _w(p, cx, cy, bc=(PER, PER), cfl=1.0, **kw):
    w = dataclasses.replace(W.tgv16(), order=p, bc_x=bc[0], bc_y=bc[1], seed=70 + p, **kw).resized(cx, cy, steps=3)
    return dataclasses.replace(w, dt=w.dt * cfl)


CASES = {
    "p1_1x1": _w(1, 1, 1), "p1_35x5": _w(1, 35, 5), "p2_17x3": _w(2, 17, 3, bc=(ZG, PER)),
    "p3_11x4": _w(3, 11, 4, bc=(PER, ZG)), "p4_9x5": _w(4, 9, 5, bc=(ZG, ZG)), "p4_2x1": _w(4, 2, 1),
    "p4_3x20": _w(4, 3, 20, cfl=2.0), "p2_20x20_far": _w(2, 20, 20, cfl=6.0), "p4_20x20_beyond": _w(4, 20, 20, cfl=12.0),
    "p2_one_population": _w(2, 19, 7, bc=(ZG, ZG), cv=1.0),
    "p3_isothermal": _w(3, 13, 3, cv=1.0, isothermal=True),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_f64_tile_against_oracle(gpu_lib, name):
    w = CASES[name]
    s, _, _ = gpu_run(w, 3, "f64")
    assert s.kernel_name == "plain_f64"
    st = s.get_state().cpu().numpy()
    for pop, ref in enumerate(H.oracle_state(w, 3)[: s.npop]):
        assert np.max(np.abs(st[pop] - ref)) <= TOL_F64 * np.max(np.abs(ref)), (name, pop)
