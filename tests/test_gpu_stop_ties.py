"""The plain form's stop test at a tolerance that equals a scenario's own step:
the one-launch solve of a small feeder and the sweep-per-launch path (the
allocation-free solve) decide alike, to the last bit."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2605_14103_gb300 import feeders as F          # noqa: E402
from paper_2605_14103_gb300 import zbus                  # noqa: E402

pytestmark = pytest.mark.gpu


def rounded(x):
    return float(x)      # of a Fraction: to nearest even


@pytest.mark.parametrize("B", [1, 40])     # both contractions of the sweep path
def test_tolerance_of_exactly_one_step(B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_14103_gb300 import build as Bd
    Bd.build()
    f = F.make_feeder(13, 3, delta_frac=0.3)
    net = zbus.Network.from_feeder(f)
    Sw, Sd = (torch.from_numpy(x).cuda() for x in F.make_scenarios(f, 40, 0.5, 1.5))
    V2, V3 = (net.solve(Sw, Sd, tol=0.0, max_iter=k)[0].cpu().numpy() for k in (2, 3))
    d = V3 - V2
    for b in range(40):
        q = [rounded(Fraction(x) ** 2 + Fraction(rounded(Fraction(y) ** 2)))
             for x, y in zip(d[b].real, d[b].imag)]
        step = float(np.sqrt(max(q)))
        lo = b if B == 1 else 0
        sw, sd = Sw[lo:lo + B], Sd[lo:lo + B]
        for tol in (step, float(np.nextafter(step, 0))):
            V, it, cv = (x.cpu().numpy() for x in net.solve(sw, sd, tol=tol))
            out = torch.empty((B, f.n), dtype=torch.complex128, device="cuda")
            it2 = torch.empty(B, dtype=torch.int32, device="cuda")
            cv2 = torch.empty(B, dtype=torch.uint8, device="cuda")
            zbus.zbus_solve_noalloc(net.handle, sw, sd, None, tol, 50, "maxabs", out, it2, cv2)
            assert np.array_equal(it, it2.cpu().numpy()), (b, tol)
            assert np.array_equal(V, out.cpu().numpy()) and np.array_equal(cv, cv2.cpu().numpy())
            # at the step itself the third map is the last
            assert it[b - lo] == (3 if tol == step else 4) or it[b - lo] < 3
    net.close()
