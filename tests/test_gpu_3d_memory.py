"""A thin 3D grid whose ghost-padded state (twice the dense one here) does not fit beside what else holds the
device's memory runs on the dense layout with the gather step, with the sum-factorised step's
results (fields to 1e-5, as the other 3D tests)."""
import numpy as np
import pytest

from .test_gpu_3d import _fields

pytestmark = pytest.mark.gpu

CELLS, P = (12, 4, 400), 3
BOX = ((0.0, 1.0), (0.0, 1.0 / 3), (0.0, 100.0 / 3))


def _run():
    from paper_1910_13918_gb300.sllbm import BC_PERIODIC, SLLBM3D
    s = SLLBM3D(cells=CELLS, order=P, box=BOX, bc=(BC_PERIODIC,) * 3, dt=0.002, tau=0.8, cv=2.5, prec="f32")
    s.precompute()
    X, Y, Z = (t.cpu().numpy() for t in s.coords())
    s.init(*_fields(X, Y, Z, BOX, 3))
    s.step(2)
    m = {k: v.cpu().numpy() for k, v in s.moments().items()}
    name = s.kernel_name
    s.close()
    return name, m


def test_the_dense_layout_where_the_padded_one_does_not_fit(gpu_lib):
    import torch
    name, ref = _run()
    assert name == "stream3d"
    torch.cuda.empty_cache()
    nv = int(np.prod([c * P for c in CELLS]))
    dense = 2 * 125 * 8 * nv                  # two buffers of (f, g) pairs
    padded = dense // nv * int(np.prod([c * P + 8 for c in CELLS]))
    keep = dense + (400 << 20)                # fields, tables and whatever the runtime takes
    assert padded > keep + (400 << 20)
    free = torch.cuda.mem_get_info()[0]
    held = torch.empty(free - keep, dtype=torch.uint8, device="cuda")
    try:
        name, m = _run()
    finally:
        del held
        torch.cuda.empty_cache()
    assert name == "gather_f32"
    for k in ref:
        assert np.max(np.abs(m[k] - ref[k])) <= 1e-5 * max(1.0, np.max(np.abs(ref[k]))), k
