"""The sum-factorised FP32 3D step at every order, on odd and ragged vertex counts, periodic and
zero-gradient, one and two populations, against the 3D oracle at the tolerances of the other 3D
tests (populations to 3e-5 of the largest deviation, density and temperature to 1e-5); time steps
whose departures leave the neighbouring cells stay in the gather step; and the state exchange,
which is exact for values that FP32 deviations hold."""
import numpy as np
import pytest

from oracle import sllbm3d as o3

from .test_gpu_3d import _gpu, _oracle

pytestmark = pytest.mark.gpu

BOX = ((0.0, 1.0), (0.0, 0.35), (0.0, 0.25))
CASES = {   # cells, p, box, periodic, dt, tau, cv, isothermal, steps
    "p1_odd": ((37, 17, 9), 1, BOX, True, 0.002, 0.8, 2.5, False, 2),
    "p2_odd_clamped": ((19, 6, 4), 2, BOX, False, 0.002, 0.8, 2.5, False, 2),
    "p3_odd": ((13, 5, 3), 3, BOX, True, 0.002, 0.7, 2.5, False, 2),
    "p3_clamped": ((12, 4, 3), 3, BOX, False, 0.002, 0.7, 2.5, False, 2),
    "p4_ragged": ((10, 4, 3), 4, BOX, True, 0.002, 0.7, 2.5, False, 2),
    "p4_odd_clamped": ((9, 3, 2), 4, BOX, False, 0.002, 0.9, 2.5, False, 2),
    "p4_isothermal": ((17, 3, 3), 4, BOX, True, 0.001, 0.9, 1.5, True, 2),
    "p3_one_population": ((12, 4, 3), 3, BOX, True, 0.002, 0.9, 1.5, False, 2),
}
FAR = {   # departures beyond the neighbouring cells, and an axis of two cells: the gather step
    "p4": ((10, 4, 2), 4, BOX, True, 0.002, 0.7, 2.5, False, 2),
    "p2_far": ((19, 6, 4), 2, BOX, True, 0.02, 0.8, 2.5, False, 1),
    "p4_far": ((9, 3, 2), 4, BOX, False, 0.01, 0.8, 2.5, False, 1),
}


@pytest.mark.parametrize("name", sorted(CASES) + sorted(FAR))
def test_tiled_orders_against_oracle(gpu_lib, name):
    case = {**CASES, **FAR}[name]
    s = _gpu(case, "f32")
    assert s.kernel_name == ("stream3d" if name in CASES else "gather_f32"), s.kernel_name
    f, g = _oracle(case)
    st = s.get_state().cpu().numpy()
    _, w = o3.d3q125()
    K = 2 * case[6] - 3
    for pop, ref in enumerate((f, g)[: s.npop]):
        lat = (w if pop == 0 else K * w)[:, None, None, None]
        scale = np.max(np.abs(ref - lat))
        assert np.max(np.abs(st[pop] - ref)) <= 3e-5 * scale, (pop, np.max(np.abs(st[pop] - ref)) / scale)
    m = s.moments()
    rho, u, th = o3.macroscopic(f, g, case[6])
    assert np.max(np.abs(m["rho"].cpu().numpy() / rho - 1)) < 1e-5
    assert np.max(np.abs(m["T"].cpu().numpy() / th - 1)) < 1e-5


@pytest.mark.parametrize("name", ["p1_odd", "p4_odd_clamped"])
def test_state_exchange_is_exact(gpu_lib, name):
    """Full populations whose deviations are FP32 values come back as they went in, and a step
    from them is the step from the state they were taken from."""
    s = _gpu(CASES[name], "f32")
    st = s.get_state()
    s.set_state(st)
    assert np.array_equal(s.get_state().cpu().numpy(), st.cpu().numpy())
    s.step(1)
    a = s.get_state().cpu().numpy()
    s.set_state(st)
    s.step(1)
    assert np.array_equal(s.get_state().cpu().numpy(), a)
