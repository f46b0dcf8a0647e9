"""The plain FP64 step on both sides of the rule that leaves its tiles for gathers on grids of few
columns or rows (tiles of 32 x 4 vertices, the rule's lines and the one-wave bound crossed from both
sides): every order, periodic and zero-gradient, against the oracle's populations after 2 steps (1e-11 of
the largest, as the other FP64 tests)."""
import numpy as np
import pytest

from paper_1910_13918_gb300 import workloads as W

from . import helpers as H
from .test_gpu_f64_tile import PER, ZG, _w
from .test_gpu_parity import TOL_F64, gpu_run

pytestmark = pytest.mark.gpu

CASES = {
    "p1_7": _w(1, 7, 2000, bc=(PER, PER)), "p1_22": _w(1, 22, 2000), "p1_row": _w(1, 15000, 1, bc=(ZG, PER)),
    "p2_8": _w(2, 4, 1000, bc=(PER, ZG)), "p2_20": _w(2, 10, 1000), "p3_13": _w(3, 4, 700, bc=(ZG, ZG)),
    "p3_18": _w(3, 6, 700), "p4_12": _w(4, 3, 500), "p4_17": _w(4, 4, 500, bc=(ZG, PER)), "p4_one_wave": _w(4, 3, 400),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_narrow_f64_against_oracle(gpu_lib, name):
    w = CASES[name]
    s, _, _ = gpu_run(w, 2, "f64")
    st = s.get_state().cpu().numpy()
    for pop, ref in enumerate(H.oracle_state(w, 2)[: s.npop]):
        assert np.max(np.abs(st[pop] - ref)) <= TOL_F64 * np.max(np.abs(ref)), (name, pop)
