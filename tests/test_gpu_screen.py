"""The mismatch test's tiers (FP32, double-float, FP64 per bus): its flags are
those of the FP64 mismatch (zbus_power_mismatch) at gates on both sides of
the scenarios' mismatches, with converged voltages moved off the fixed point
by a loose stop rule, on three- and partial-phase feeders and in every form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

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


@pytest.mark.parametrize("form", ["fp16_scaled", "bf16x2", "tree"])
@pytest.mark.parametrize("N,B,lateral,tol", [(13, 5, 0.0, 1e-4), (60, 33, 0.3, 1e-5),
                                             (128, 257, 0.0, 1e-6), (400, 64, 0.0, 1e-5)])
def test_flags_are_those_of_the_fp64_mismatch(form, N, B, lateral, tol):
    if lateral:
        f = F.make_partial_feeder(N, 11, lateral_frac=lateral, delta_frac=0.4)
        Sw, Sd = F.make_partial_scenarios(f, B, 0.5, 1.2)
    else:
        f = F.make_feeder(N, 500 + N, delta_frac=0.4)
        Sw, Sd = F.make_scenarios(f, B, 0.5, 1.2)
    Sw, Sd = torch.from_numpy(Sw).cuda(), torch.from_numpy(Sd).cuda()
    net = zbus.Network.from_feeder(f)
    kw = dict(tol=tol, precision=form, max_correction=0)
    V, it, cv = net.solve(Sw, Sd, mismatch_tol=1e3, **kw)
    assert cv.all()
    mm = net.power_mismatch(V, Sw, Sd).cpu().numpy()
    # gates on the tiers' side of 5e-7, between the scenarios' mismatches
    gates = [g for g in np.quantile(mm, [0.1, 0.5, 0.9]) * 1.000001 if g >= 5e-7]
    for gate in gates + [1e-6, 1e-5, 1e-4, 1e-2]:
        clear = np.abs(mm / gate - 1.0) > 1e-9      # rounding of two FP64 orders of sums
        V2, it2, cv2 = net.solve(Sw, Sd, mismatch_tol=gate, **kw)
        assert torch.equal(V2, V) and torch.equal(it2, it)
        assert np.array_equal(cv2.cpu().numpy()[clear] != 0, (mm <= gate)[clear]), gate
    net.close()
