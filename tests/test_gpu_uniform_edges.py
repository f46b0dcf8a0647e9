"""Uniform grids at the edges of the fused kernel's range: periodic axes whose vertex counts are no
multiple of 4 (down to three cells), and the warp-per-vertex fix-up of the vertices next to
zero-gradient boundaries with every option it carries (storage, Prandtl number, one population,
the isothermal equilibrium, the moments epilogue).  FP32 against the oracle at the tolerances of
the other parity tests: 1e-5 after one step, 1e-4 after 30.  On states larger than the L2 (over
64 MB) the edge-tile launch takes those vertices: one step against the plain FP64 step from the
same state, every value within 2e-6 (about 30 FP32 roundings of values below 1)."""
import dataclasses

import numpy as np
import pytest

from paper_1910_13918_gb300 import workloads as W

from . import helpers as H
from .test_gpu_parity import TOL_1, TOL_100, gpu_run

pytestmark = pytest.mark.gpu

ZG, PER = W.ZERO_GRADIENT, W.PERIODIC


def _tgv(p, cells_x, cells_y, bc=(PER, PER), **kw):
    w = dataclasses.replace(W.tgv16(), order=p, bc_x=bc[0], bc_y=bc[1], seed=40 + p, **kw)
    return w.resized(cells_x, cells_y, steps=30)


CASES = {
    "p1_three_cells": _tgv(1, 3, 3), "p1_37": _tgv(1, 37, 9), "p2_three_cells": _tgv(2, 3, 5),
    "p2_34": _tgv(2, 17, 4), "p3_33": _tgv(3, 11, 5), "p3_43": _tgv(3, 43, 7), "p3_81": _tgv(3, 27, 3),
    "p3_mixed": _tgv(3, 15, 5, bc=(PER, ZG)),
    "p1_clamped": _tgv(1, 33, 7, bc=(ZG, ZG)), "p2_clamped_x": _tgv(2, 16, 4, bc=(ZG, PER)),
    "p3_clamped": _tgv(3, 14, 5, bc=(ZG, ZG)), "p4_clamped_pr": _tgv(4, 9, 4, bc=(ZG, ZG), pr=0.75),
    "p2_clamped_one_population": _tgv(2, 13, 6, bc=(ZG, ZG), cv=1.0),
    "p4_clamped_isothermal": _tgv(4, 9, 5, bc=(ZG, ZG), cv=1.0, isothermal=True),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("nsteps,tol", [(1, TOL_1), (30, TOL_100)])
def test_edges_f32(gpu_lib, name, nsteps, tol):
    w = CASES[name]
    s, gpu, _ = gpu_run(w, nsteps, "f32")
    assert s.kernel_name == "uniform_fused", s.kernel_name
    err = H.field_errors(gpu, H.oracle_run(w, nsteps), w.velocity_scale)
    assert max(err.values()) <= tol, (name, err)


@pytest.mark.parametrize("name", ["p3_33", "p3_mixed", "p4_clamped_pr", "p2_clamped_x"])
def test_edges_bf16(gpu_lib, name):
    w = CASES[name]
    s, gpu, _ = gpu_run(w, 5, "bf16")
    assert s.kernel_name == "uniform_fused", s.kernel_name
    err = H.field_errors(gpu, H.oracle_run(w, 5), w.velocity_scale)
    assert max(err.values()) <= 2e-2, (name, err)


@pytest.mark.parametrize("name", ["p3_clamped", "p4_clamped_pr", "p2_clamped_one_population"])
def test_edges_moments_epilogue(gpu_lib, name):
    """The moments a step writes are those of its state (the collision conserves them)."""
    import torch
    w = CASES[name]
    s, _, _ = gpu_run(w, 2, "f32")
    mom = torch.empty((4, s.ny, s.nx), dtype=torch.float32, device="cuda")
    s.step_moments(mom)
    m = s.moments()
    for k, key in enumerate(("rho", "u", "v", "T")):
        a, b = mom[k].cpu().numpy().astype(np.float64), m[key].cpu().numpy().astype(np.float64)
        assert np.max(np.abs(a - b)) <= 3e-6 * max(1.0, np.max(np.abs(b))), (name, key)


LARGE = {   # over 335,544 vertices: 50 FP32 values a vertex are more than 64 MB
    "p1_clamped": _tgv(1, 600, 577, bc=(ZG, ZG)), "p2_clamped_y": _tgv(2, 301, 300, bc=(PER, ZG)),
    "p3_clamped_x": _tgv(3, 197, 200, bc=(ZG, PER)), "p3_clamped_pr": _tgv(3, 200, 191, bc=(ZG, ZG), pr=0.75),
    "p4_clamped": _tgv(4, 151, 147, bc=(ZG, ZG)), "p4_strip": _tgv(4, 20000, 4, bc=(ZG, ZG)),
}


@pytest.mark.parametrize("name", sorted(LARGE))
def test_edge_tiles_against_the_plain_step(gpu_lib, name):
    from paper_1910_13918_gb300.sllbm import SLLBM
    w = LARGE[name]
    a, b = SLLBM.from_workload(w, prec="f32"), SLLBM.from_workload(w, prec="f64")
    for s in (a, b):
        s.precompute()
    x, y = (t.cpu().numpy() for t in a.coords())
    a.init(*w.fields(x, y, perturb=True))
    lat = np.outer(*[np.array(H.o.d1q5()[1])] * 2).reshape(-1)
    full = a.get_state().double()
    for k, c in enumerate((1.0, 2 * w.cv - 2)):
        full[k] += c * full.new_tensor(lat)[:, None, None]
    b.set_state(full)
    a.step(1)
    b.step(1)
    got, ref = a.get_state().double(), b.get_state()
    for k, c in enumerate((1.0, 2 * w.cv - 2)):
        ref[k] -= c * ref.new_tensor(lat)[:, None, None]
    err = float((got - ref).abs().max())
    assert (a.kernel_name, a.launches_per_step) == ("uniform_fused", 2)
    assert err <= 2e-6, (name, err)
