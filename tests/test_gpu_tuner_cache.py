"""Cache files that earlier versions of the tuner wrote (GPU)."""

import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import sys; sys.path.insert(0, %r)
import numpy as np
import paper_2204_03775_gb300 as wsb
wsb.load_library(build_if_missing=True)
h = wsb.ws_create(130, 40, 30, 10.0, 1e-3)
wsb.ws_set_velocity(h, np.full((30, 40, 130), 2000.0, np.float32))
n0 = wsb.ws_launch_count(h)
t = wsb.ws_autotune(h)
print(*t, wsb.ws_launch_count(h) - n0)
""" % ROOT


def test_tunings_of_another_kernel_version_are_not_taken(tmp_path):
    """A line without the kernel's version, as the file held before the
    streaming kernel was rewritten, names a tiling that was never timed on
    this one: the grid is tuned again, and the new line is used from then on."""
    path = tmp_path / "tune.txt"
    old = "%s|0|130|40|30|32|8|3" % torch.cuda.get_device_name(0)
    path.write_text(old + "\n")
    env = dict(os.environ, WS_TUNE_CACHE=str(path))
    runs = []
    for _ in range(2):
        r = subprocess.run([sys.executable, "-c", CODE], env=env, capture_output=True, text=True,
                           timeout=300)
        assert r.returncode == 0, r.stderr
        runs.append(list(map(int, r.stdout.split())))
    assert runs[0][3] > 0 and runs[1][3] == 0, runs
    assert runs[0][:3] == runs[1][:3]
    lines = [line for line in path.read_text().splitlines() if line != old]
    assert len(lines) == 1 and lines[0].split("|")[1:5] == ["0", "130", "40", "30"]
