"""State exchange of long narrow grids: few columns and many rows (also more rows than a grid dimension
holds), few rows and many columns, and the widths at which the conversion changes its blocks, for
both layouts ((f, g) pairs and single planes) and every storage.  The state handed in comes back as
it was, through the device and the host path, and every vertex carries its own values."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_1910_13918_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (2, 3000), (3, 70001), (5, 131), (17, 300), (32, 33), (33, 31), (127, 9), (128, 5), (129, 6), (257, 3), (9000, 1)]


@pytest.mark.parametrize("prec,velset", [("f32", "d2q25"), ("bf16", "d2q25"), ("f64", "d2q25"), ("f32", "d2q9"), ("bf16", "d2q9")])
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_round_trip(gpu_lib, nx, ny, prec, velset):
    from paper_1910_13918_gb300.sllbm import SLLBM
    cv = 1.0 if velset == "d2q9" else 2.5
    w = dataclasses.replace(W.tgv16(), order=1, cv=cv, isothermal=velset == "d2q9", velset=velset).resized(nx, ny)
    s = SLLBM.from_workload(w, prec=prec)
    s.precompute()
    shape = (s.npop, s.nq, ny, nx)
    bits = {2: torch.int16, 4: torch.int32, 8: torch.int64}[torch.empty(0, dtype=s.state_dtype).element_size()]
    st = torch.arange(int(np.prod(shape)), device="cuda").to(bits).reshape(shape)   # a pattern of its own per value
    s.set_state(st)
    assert torch.equal(s.get_state().view(bits), st)
    host = st.cpu().view(torch.uint8).numpy().reshape(-1)
    out = np.empty_like(host)
    s.step_host(host, out, 0)
    assert np.array_equal(out, host)
