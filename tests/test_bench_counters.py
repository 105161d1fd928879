"""What bench.py makes of the kernel-class counts (CPU only)."""

import importlib.util
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_work_done_inside_another_kernel_is_not_a_launch(monkeypatch):
    monkeypatch.setenv("CUDA_DEVICE_MAX_CONNECTIONS", "8")  # bench.py sets a default; put back afterwards
    spec = importlib.util.spec_from_file_location("bench_for_counters", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    # class: (counted, timed, ms), with every class timed; B~_q ("g3") is done by the SVD kernel
    profile = {"theta": (100, 100, 1.0), "svd": (100, 100, 5.0), "g3": (100, 0, 0.0), "gate1": (0, 0, 0.0)}
    assert bench.own_launches({"theta": (50, 0, 0.0), "svd": (50, 0, 0.0), "g3": (50, 0, 0.0)}, profile) == 100
    # with its own kernel (the FP32 SVD, tensor cores) it counts
    profile["g3"] = (100, 100, 0.5)
    assert bench.own_launches({"theta": (50, 0, 0.0), "svd": (50, 0, 0.0), "g3": (50, 0, 0.0)}, profile) == 150
