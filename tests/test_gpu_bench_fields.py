"""The benchmark compares its forms at the same step: the fields that a form is judged by are those after
the warm-up and timed steps, whether its context is kept (and takes more steps for other timings) or not."""
import argparse
import importlib.util
import os

import pytest

from . import helpers as H

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fields_of_a_kept_form(gpu_lib):
    import torch
    spec = importlib.util.spec_from_file_location("bench_module", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    w = H.small_workloads()["tgv256"]
    args = argparse.Namespace(steps=4, warmup=3, repeats=2)
    kept, left = (bench.measure(w, "f32", args, torch.cuda.Stream(), [0, 5], keep=k) for k in (True, False))
    assert torch.equal(kept["final"], left["final"])
    assert kept["info"]["mass_after"] == left["info"]["mass_after"]
    assert kept["info"]["ms_per_step_with_moments"] > 0
