"""The bounds-check build checks every population element that a step touches: a window of
the buffers is declared outside (the memory stays valid), and a step must count and skip
every access into it (tests/bounds_window_cases.py, in a child process)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2510_14712_gb300")
HERE = os.path.dirname(os.path.abspath(__file__))


def test_every_access_into_a_hidden_window_is_counted_and_skipped():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14712_gb300 import build
    env = dict(os.environ, LBM_LIBRARY=build.build(bounds_check=True))
    r = subprocess.run([sys.executable, os.path.join(HERE, "bounds_window_cases.py")], env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    assert "windows: 0 of" in r.stdout, r.stdout[-4000:]
