"""The DRAM traffic that bench.py reports from stored captures is never less than what the step has to move:
the state read once and written once (8 B an update)."""
import importlib.util
import os

import pytest

from paper_1910_13918_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_spec = importlib.util.spec_from_file_location("bench_module", os.path.join(ROOT, "bench.py"))
bench = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(bench)


@pytest.mark.parametrize("key", sorted(bench.NCU_TRAFFIC), ids=lambda k: k[1])
def test_traffic_covers_the_algorithmic_bytes(key):
    _, name, prec = key
    w = {w.name: w for w in (bench._workload(n) for n in ("riemann_paper", "riemann_paper512", "tgv256"))}[name]
    least = w.updates_per_step * bench.bytes_per_update(w, prec, "uniform_fused")
    assert least <= bench.NCU_TRAFFIC[key] <= 1.25 * least
