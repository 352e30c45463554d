"""Batches above one 32-scenario tile of feeders of at most 96 padded unknowns:
the one-launch solve gives the bits of the sweep kernels (which the profile
mode launches), whatever the batch."""
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


def bits(V):
    return V.view(torch.float64).view(torch.int64)


@pytest.mark.parametrize("N,rule", [(13, "maxabs"), (33, "summag")])
def test_bits_of_the_sweep_kernels(N, rule):
    f = F.make_feeder(N, 40 + N, delta_frac=0.4, mult_hi=1.5)
    Sw, Sd = (torch.from_numpy(x).cuda() for x in F.make_scenarios(f, 2049, 0.5, 1.5))
    Sw[7] *= 500.0
    net = zbus.Network.from_feeder(f)
    whole = net.solve(Sw, Sd, rule=rule, profile=True)
    for B in (33, 2049):
        V, it, cv = net.solve(Sw[:B].contiguous(), Sd[:B].contiguous(), rule=rule)
        assert torch.equal(bits(V), bits(whole[0][:B]))
        assert torch.equal(it, whole[1][:B]) and torch.equal(cv, whole[2][:B])
    net.close()
