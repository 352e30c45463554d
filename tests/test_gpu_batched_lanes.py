"""Batched solve on a caller's stream: feeders are admitted and collected on
several streams, which wait for the caller's and which it waits for."""
import numpy as np
import pytest
import torch

from paper_2605_14103_gb300 import feeders as F
from paper_2605_14103_gb300 import zbus

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["fp16_scaled", "tree"])
@pytest.mark.parametrize("items", [1, 2, 4, 5, 9])
def test_lanes_are_ordered_with_the_callers_stream(items, mode):
    """Loads made just before the call and overwritten just after it on the
    same stream, outputs copied on it: the results are a single solve's."""
    fs = [F.make_feeder(20 + 37 * k, 60 + k, delta_frac=0.4) for k in range(items)]
    nets = [zbus.Network.from_feeder(f) for f in fs]
    host = [[torch.from_numpy(np.ascontiguousarray(a)).cuda()
             for a in F.make_scenarios(f, 200 - 17 * k, 0.8, 1.2)] for k, f in enumerate(fs)]
    alone = [net.solve(*x, precision=mode) for net, x in zip(nets, host)]
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(2):
        with torch.cuda.stream(st):
            loads = [tuple(2.0 * (0.5 * a) for a in x) for x in host]
            outs = zbus.solve_batched(nets, loads, precision=mode)
            for pair in loads:
                for a in pair:
                    a.fill_(3.0)
            got = [tuple(a.clone() for a in o) for o in outs]
            for o in outs:
                for a in o:
                    a.zero_()
        st.synchronize()
        for (V, it, cv), (V1, it1, cv1) in zip(got, alone):
            assert torch.equal(it, it1) and torch.equal(cv, cv1)
            assert (V - V1).abs().max().item() <= 1e-12
    for net in nets:
        net.close()
