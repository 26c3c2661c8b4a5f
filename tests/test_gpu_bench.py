"""The benchmark's JSON line on small batches of the 2,000-bus grid: what a reader of
the line relies on, whichever kernels the batch and the precision select."""
import importlib.util
import pathlib
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lu,batch", [("fp64", 96), ("fp32", 96), ("fp32", 640)])
def test_line_counts_its_launches(lu, batch, monkeypatch):
    import paper_2101_02270_gb300 as pf
    spec = importlib.util.spec_from_file_location("bench", pathlib.Path(__file__).parent.parent / "bench.py")
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    monkeypatch.setattr(sys, "argv", ["bench.py", "--no-oracle", "--no-cpu-baseline"])
    line = bench.measure_mesh(bench.parse_args(), pf, "mesh2000_b10k", lu, 1, 3, torch.device("cuda", 0), batch=batch,
                              with_cpu=False, e2e=False)
    assert type(line["gpu_launches"]) is int and line["gpu_launches"] > 0
    assert type(line["roofline"]["launches"]) is int and line["roofline"]["achieved"] > 0
    assert line["converged"] == batch
