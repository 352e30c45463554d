"""The digit sweeps (csrc/split.cu) on a device too full for the scratch of a
whole batch: passes of fewer scenarios with the same bits, not another method
(tests/split_passes_run.py)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_a_batch_in_passes_keeps_its_bits():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_14103_gb300 import build as B
    env = dict(os.environ, ZBUS_LIB=B.build(checked=True))
    r = subprocess.run([sys.executable, os.path.join(HERE, "split_passes_run.py")], env=env,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "passes ok" in r.stdout
