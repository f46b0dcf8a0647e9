"""The forward pass of a rollout takes every step once, in segments that end where a checkpoint is
kept, for any checkpoint interval: on the CPU, with a simulation that counts its steps."""
import types

import pytest
import torch

from paper_1910_13918_gb300.autograd import SLLBMRollout


class _Sim:
    _stream = None

    def init(self, *fields):
        self.n, self.calls = 0, []

    def step(self, n=1):
        assert n > 0
        self.n += n
        self.calls.append(n)

    def get_state(self):
        return self.n

    def moments(self, sums=True):
        return {"rho": torch.tensor([float(self.n)])}


@pytest.mark.parametrize("nsteps,k,kept,calls", [
    (10, 5, [0, 5], [5, 5]), (10, 3, [0, 3, 6, 9], [3, 3, 3, 1]), (2, 20, [0], [2]), (3, 1, [0, 1, 2], [1, 1, 1]),
    (10, -3, [0, 3, 6, 9], [3, 3, 3, 1]), (0, 5, [0], []), (0, 0, [0], []),
])
def test_forward_segments(monkeypatch, nsteps, k, kept, calls):
    import contextlib
    monkeypatch.setattr(torch.cuda, "stream", lambda s: contextlib.nullcontext())
    sim, ctx = _Sim(), types.SimpleNamespace(save_for_backward=lambda *t: None)
    t = torch.zeros(1)
    rho = SLLBMRollout.forward(ctx, t, t, sim, t, t, nsteps, k)
    assert float(rho) == nsteps and sim.calls == calls
    assert ctx.checkpoints == {n: n for n in kept}


def test_an_interval_of_zero_is_refused(monkeypatch):
    import contextlib
    monkeypatch.setattr(torch.cuda, "stream", lambda s: contextlib.nullcontext())
    t = torch.zeros(1)
    with pytest.raises(ZeroDivisionError):
        SLLBMRollout.forward(types.SimpleNamespace(save_for_backward=lambda *t: None), t, t, _Sim(), t, t, 4, 0)
