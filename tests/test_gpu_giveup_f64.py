"""The bounded waits of the plain FP64 form's contraction (csrc/split.cu) give
up without a fault in the checked build, as those of the mixed forms do
(tests/giveup_f64_run.py)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_fp64_contraction_gives_up_and_recovers():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_14103_gb300 import build as B
    env = dict(os.environ, ZBUS_LIB=B.build(checked=True))
    r = subprocess.run([sys.executable, os.path.join(HERE, "giveup_f64_run.py")], env=env,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "giveup ok" in r.stdout


def test_device_status_is_the_networks_last_solve():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_14103_gb300 import build as B
    env = dict(os.environ, ZBUS_LIB=B.build(checked=True))
    r = subprocess.run([sys.executable, os.path.join(HERE, "device_status_run.py")], env=env,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "status ok" in r.stdout
