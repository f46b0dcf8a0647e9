"""The edge-tile launch of the fused uniform step, over all it carries: FP32 and BF16 storage, Prandtl
number, one population, the isothermal equilibrium, the moments epilogue, several steps a call, on states
larger than the L2 (64 MB) and on long thin grids with more than 2,000 vertices next to
zero-gradient boundaries (and just below that, where the fix-up kernel takes them).  One step against the plain
FP64 step from the same state: FP32 within 2e-6 (about 30 FP32 roundings of values below 1), BF16 within
that and one BF16 spacing, 2^-8, of the value."""
import numpy as np
import pytest

from . import helpers as H
from .test_gpu_uniform_edges import LARGE, PER, ZG, _tgv

pytestmark = pytest.mark.gpu

THIN = {   # off the cell pattern: about one row or column a clamped side
    "p1_thin": _tgv(1, 1200, 7, bc=(ZG, ZG)), "p1_below": _tgv(1, 900, 7, bc=(PER, ZG)), "p2_thin": _tgv(2, 700, 4, bc=(PER, ZG)),
    "p2_tall": _tgv(2, 5, 600, bc=(ZG, PER)), "p3_thin": _tgv(3, 500, 3, bc=(ZG, ZG)), "p3_pr": _tgv(3, 400, 4, bc=(PER, ZG), pr=0.75),
    "p4_thin": _tgv(4, 300, 3, bc=(ZG, ZG)), "p4_one_population": _tgv(4, 300, 3, bc=(PER, ZG), cv=1.0),
    "p2_isothermal": _tgv(2, 700, 4, bc=(ZG, ZG), cv=1.0, isothermal=True),
}
LARGE_BF16 = {   # over 671,088 vertices: 50 BF16 values a vertex are more than 64 MB
    "p1": _tgv(1, 850, 820, bc=(ZG, ZG)), "p2_y": _tgv(2, 431, 400, bc=(PER, ZG)), "p3": _tgv(3, 281, 270, bc=(ZG, ZG)),
    "p3_pr_x": _tgv(3, 281, 270, bc=(ZG, PER), pr=0.75), "p4": _tgv(4, 207, 205, bc=(ZG, ZG)),
    "p4_one_population": _tgv(4, 290, 292, bc=(ZG, ZG), cv=1.0),
}


def _pair(w, prec):
    """The fused context and a plain FP64 one, both at the fused one's state."""
    from paper_1910_13918_gb300.sllbm import SLLBM
    a, b = SLLBM.from_workload(w, prec=prec), SLLBM.from_workload(w, prec="f64")
    for s in (a, b):
        s.precompute()
    x, y = (t.cpu().numpy() for t in a.coords())
    a.init(*w.fields(x, y, perturb=True))
    full = a.get_state().double()
    for k, c in enumerate((1.0, 2 * w.cv - 2)[: a.npop]):
        full[k] += c * _lattice(full)
    b.set_state(full)
    return a, b


def _lattice(t):
    return t.new_tensor(np.outer(*[np.array(H.o.d1q5()[1])] * 2).reshape(-1))[:, None, None]


def _check_step(w, prec):
    a, b = _pair(w, prec)
    a.step(1)
    b.step(1)
    got, ref = a.get_state().double(), b.get_state()
    for k, c in enumerate((1.0, 2 * w.cv - 2)[: a.npop]):
        ref[k] -= c * _lattice(ref)
    bound = 2e-6 + (2.0 ** -8 * ref.abs() if prec == "bf16" else 0.0)
    assert a.kernel_name == "uniform_fused"
    assert bool(((got - ref).abs() <= bound).all()), float((got - ref).abs().max())


@pytest.mark.parametrize("name", sorted(THIN))
@pytest.mark.parametrize("prec", ["f32", "bf16"])
def test_thin_grids(gpu_lib, name, prec):
    _check_step(THIN[name], prec)


@pytest.mark.parametrize("name", sorted(LARGE_BF16))
def test_large_grids_bf16(gpu_lib, name):
    _check_step(LARGE_BF16[name], "bf16")


EPILOGUE = {**{k: (LARGE[k], "f32") for k in ("p2_clamped_y", "p3_clamped_pr", "p4_strip")},
            **{k: (THIN[k], "f32") for k in ("p1_thin", "p2_tall", "p3_pr", "p4_one_population")},
            "bf16_p3": (LARGE_BF16["p3"], "bf16")}


@pytest.mark.parametrize("name", sorted(EPILOGUE))
def test_moments_epilogue(gpu_lib, name):
    """Every vertex's moments are written, and are those of the state the step makes (to FP32, or
    the BF16 rounding of the stored state)."""
    import torch
    w, prec = EPILOGUE[name]
    a, _ = _pair(w, prec)
    a.step(1)
    buf = torch.full((4, a.ny, a.nx), float("nan"), dtype=torch.float32, device="cuda")
    a.step_moments(buf)
    m = a.moments()
    assert bool(torch.isfinite(buf).all())
    for k, key in enumerate(("rho", "u", "v", "T")):
        err = float((buf[k].double() - m[key].double()).abs().max())
        assert err <= (3e-6 if prec == "f32" else 3e-2) * max(1.0, float(m[key].abs().max())), (key, err)


@pytest.mark.parametrize("name", ["large", "thin", "tall", "bf16"])
def test_steps_in_one_call_equal_single_steps(gpu_lib, name):
    import torch
    w, prec = {"large": (LARGE["p3_clamped_x"], "f32"), "thin": (THIN["p3_thin"], "f32"), "tall": (THIN["p2_tall"], "f32"),
               "bf16": (THIN["p4_thin"], "bf16")}[name]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        from paper_1910_13918_gb300.sllbm import SLLBM
        out = []
        for calls in ([7, 4], [1] * 11):
            s = SLLBM.from_workload(w, prec=prec, stream=stream)
            s.precompute()
            x, y = (t.cpu().numpy() for t in s.coords())
            s.init(*w.fields(x, y, perturb=True))
            for n in calls:
                s.step(n)
            out.append(s.get_state().contiguous().view(torch.uint8))
        same = torch.equal(*out)
    stream.synchronize()
    assert same
