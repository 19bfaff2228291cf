"""A step that gives up its bounded wait leaves part of the new state unwritten
(LBM_FLAG_INCOMPLETE): the handle or the batch's instance refuses to step on and to give
fields or populations until it is initialised again.  The flag is raised by a debug entry
of the bounds-check build, in a child process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2510_14712_gb300")
HERE = os.path.dirname(os.path.abspath(__file__))


def test_incomplete_state_is_refused():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14712_gb300 import build
    env = dict(os.environ, LBM_LIBRARY=build.build(bounds_check=True))
    r = subprocess.run([sys.executable, os.path.join(HERE, "incomplete_cases.py")], env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0 and "incomplete ok" in r.stdout, r.stderr[-3000:]
