"""How vqe_eval_batch feeds its streams: counted by device.

Host code only.  Up to eight streams of a device, its default hardware queues,
are fed gate by gate; those of a device with more get runs of gates.  Streams
on another device do not count.
"""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2303_03681_gb300 import build as _build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("rule") / "batch_rule.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-I", _build.CSRC,
                    os.path.join(HERE, "native", "batch_rule.cu"), _build.build(), "-o", lib,
                    "-Xlinker", "-rpath," + os.path.dirname(_build.LIB)], check=True)
    return ctypes.CDLL(lib)


@pytest.mark.parametrize("devices,by_gate", [
    ([0] * 8, [1] * 8),
    ([0] * 9, [0] * 9),
    ([0, 1] * 8, [1] * 16),                    # sixteen streams, eight on each device
    ([0] * 9 + [1] * 3, [0] * 9 + [1] * 3),
    ([], []),
])
def test_streams_count_on_their_own_device(rule, devices, by_gate):
    dev = np.array(devices, np.int32)
    out = np.zeros(max(1, len(devices)), np.int8)
    rule.gate_by_gate_streams(ctypes.c_void_p(dev.ctypes.data), len(devices), ctypes.c_void_p(out.ctypes.data))
    assert list(out[: len(devices)]) == by_gate
