"""The mismatch test of the mixed forms (k_screen) on buses its FP32 tier cannot
bound: a delta branch whose voltage has cancelled, and loads outside the range
of FP32.  Flags and voltages are those of the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import zbus_oracle as O                      # noqa: E402
from paper_2605_14103_gb300 import feeders as F          # noqa: E402
from paper_2605_14103_gb300 import zbus                  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_14103_gb300 import build as B
    B.build()
    zbus.lib()


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def check(f, v_slack, Sw, Sd, form):
    net = zbus.Network(f.n_total, f.Y_row, f.Y_col, f.Y_val, f.slack_idx, v_slack)
    ref = O.solve_coo(f.n_total, f.Y_row, f.Y_col, f.Y_val, f.slack_idx, v_slack, Sw, Sd)
    V, it, cv = net.solve(dev(Sw), dev(Sd), precision=form)
    mm = net.power_mismatch(V, dev(Sw), dev(Sd)).cpu().numpy()
    V, cv = V.cpu().numpy(), cv.cpu().numpy()
    assert np.array_equal(cv, ref["converged"])
    ok = cv == 1
    assert (mm[ok] <= 1e-6).all()
    assert np.abs(V[ok] - ref["V"][ok]).max(initial=0.0) <= 1e-6
    net.close()
    return ok


@pytest.mark.parametrize("form", ["fp16_scaled", "tree"])
def test_branch_voltage_that_cancels(form):
    """Phases a and b of the slack 2^-14 apart: the branch ab of every bus has
    a voltage of 2^-14, its load's current is an ordinary one."""
    f = F.make_feeder(13, 5)
    B = 33
    rng = np.random.default_rng(5)
    vs = np.array([1.0, 1.0 + 2.0 ** -14, np.exp(2j * np.pi / 3)], dtype=np.complex128)
    Sw = np.zeros((B, f.n), dtype=np.complex128)
    Sd = np.zeros((B, f.n), dtype=np.complex128)
    Sw[:, 2::3] = rng.uniform(0.5, 1.5, size=(B, f.n // 3)) * (0.02 + 0.01j)
    Sd[:, 0::3] = rng.uniform(0.5, 1.5, size=(B, f.n // 3)) * 2.0 ** -35
    assert check(f, vs, Sw, Sd, form).all()


@pytest.mark.parametrize("form", ["fp16_scaled", "tree"])
def test_loads_outside_the_range_of_fp32(form):
    """Loads of 1e-60 (zero in FP32) converge, one of 1e60 (infinite) does not."""
    f = F.make_feeder(13, 6, delta_frac=0.5)
    Sw, Sd = F.make_scenarios(f, 33, 0.8, 1.2)
    Sw[3:9] *= 1e-60
    Sd[3:9] *= 1e-60
    Sw[20, 4] = 1e60
    ok = check(f, f.v_slack, Sw, Sd, form)
    assert ok[:20].all() and not ok[20] and ok[21:].all()
