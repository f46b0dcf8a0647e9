"""The whole-cell D2Q9 kernel (periodic uniform grids) at every order, on ragged and odd vertex
counts, in FP32 against the oracle at the tolerances of the other D2Q9 tests (1e-5 after one step,
1e-4 after 30) and with BF16 storage (3e-2 after 5)."""
import dataclasses

import pytest

from paper_1910_13918_gb300 import workloads as W

from . import helpers as H
from .test_gpu_parity import TOL_1, TOL_100, gpu_run

pytestmark = pytest.mark.gpu


def _w(p, cx, cy):
    w = W.tgv_moving(16, 0.05, "d2q9")
    return dataclasses.replace(w, order=p, nx_cells=cx, ny_cells=cy, dt=0.25 * w.dt, seed=60 + p)


CASES = {"p1_33x3": _w(1, 33, 3), "p1_5x37": _w(1, 5, 37), "p2_34x6": _w(2, 17, 3), "p2_66x22": _w(2, 33, 11),
         "p3_9x9": _w(3, 3, 3), "p3_33x15": _w(3, 11, 5), "p3_99x27": _w(3, 33, 9), "p4_12x12": _w(4, 3, 3),
         "p4_36x20": _w(4, 9, 5), "p4_68x32": _w(4, 17, 8)}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("nsteps,tol", [(1, TOL_1), (30, TOL_100)])
def test_cells_f32(gpu_lib, name, nsteps, tol):
    w = CASES[name]
    s, gpu, _ = gpu_run(w, nsteps, "f32")
    assert s.kernel_name == "d2q9"
    err = H.field_errors(gpu, H.oracle_run(w, nsteps), w.velocity_scale)
    assert max(err.values()) <= tol, (name, err)


@pytest.mark.parametrize("name", ["p3_33x15", "p4_36x20", "p1_5x37"])
def test_cells_bf16(gpu_lib, name):
    w = CASES[name]
    _, gpu, _ = gpu_run(w, 5, "bf16")
    err = H.field_errors(gpu, H.oracle_run(w, 5), w.velocity_scale)
    assert max(err["rho"], err["u"], err["v"]) < 3e-2, err
