"""Host threads that solve networks of different sizes with the plain FP64 form
at the same time, each on its own stream: every launch is accepted and every
result is that of a solve by itself."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2605_14103_gb300 import feeders as F          # noqa: E402
from paper_2605_14103_gb300 import zbus                  # noqa: E402

pytestmark = pytest.mark.gpu


def test_two_sizes_at_once(monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_14103_gb300 import build as B
    B.build()
    monkeypatch.setenv("ZBUS_NO_GRAPH", "1")    # every sweep is a launch of the host
    jobs = []
    for N in (690, 1100):       # shared memory of 33 and 53 KB a block
        f = F.make_feeder(N, N)
        net = zbus.Network.from_feeder(f)
        Sw = torch.from_numpy(F.make_scenarios(f, 2, 0.8, 1.2)[0]).cuda()
        want = [x.cpu().numpy() for x in net.solve(Sw, None)]
        jobs.append((net, Sw, want, torch.cuda.Stream()))
    torch.cuda.synchronize()
    wrong = []

    def work(net, Sw, want, st):
        try:
            torch.cuda.set_device(0)
            with torch.cuda.stream(st):
                for _ in range(60):
                    got = net.solve(Sw, None, stream=st)
                    st.synchronize()
                    for x, y in zip(got, want):
                        assert np.array_equal(x.cpu().numpy(), y)
        except Exception as e:   # noqa: BLE001 - reported by the main thread
            wrong.append(repr(e))

    ts = [threading.Thread(target=work, args=j) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not wrong, wrong
    for net, *_ in jobs:
        net.close()
