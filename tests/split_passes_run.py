"""Child process of tests/test_gpu_split_passes.py, in the checked build: where
the device does not hold the digit sweeps' scratch of a whole batch
(ZBUS_CHECKED_SPLIT_BYTES stands in for it), the batch runs in passes of fewer
scenarios, and the bits stay.  Prints "passes ok" on success."""
import os
import sys

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from paper_2605_14103_gb300 import feeders as F          # noqa: E402
from paper_2605_14103_gb300 import zbus                  # noqa: E402


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def limit(n, rows):
    """Bytes that hold the scratch of `rows` scenarios and not of 128 more
    (22 planes of halves and of 32-bit integers, the operand, a few words)."""
    if rows is None:
        os.environ.pop("ZBUS_CHECKED_SPLIT_BYTES", None)
    else:
        per = 22 * (2 * ((n + 63) // 64 * 64) + 4 * ((n + 7) // 8 * 8)) + 16 * n + 20
        os.environ["ZBUS_CHECKED_SPLIT_BYTES"] = str((rows + 64) * per)


def main():
    flag, _ = zbus.zbus_checked_status()
    assert flag == 1, "not the checked build"
    f = F.make_feeder(50, 3, delta_frac=0.3)
    for B, rows in ((300, 128), (513, 256), (256, 128)):   # two passes and a rest, or none
        Sw, Sd = (dev(x) for x in F.make_scenarios(f, B, 0.5, 1.5, seed=B))
        Sw[B // 2] = 0     # stops after one map, in a pass of its own length
        Sd[B // 2] = 0
        G = torch.from_numpy(np.random.default_rng(B).normal(size=(B, f.n)) * (1 + 0.5j)).cuda()

        def both(net, rule):
            V, it, cv = net.solve(Sw, Sd, rule=rule)
            return [V, it, cv, *net.solve_adjoint(V, G, Sw, Sd)]

        for rule in ("maxabs", "summag"):
            limit(f.n, None)
            one = zbus.Network.from_feeder(f)
            want = [x.cpu().numpy() for x in both(one, rule)]
            limit(f.n, rows)
            few = zbus.Network.from_feeder(f)
            for _ in range(2):
                for x, y in zip(both(few, rule), want):
                    assert np.array_equal(x.cpu().numpy(), y), (B, rows, rule)
            # warm starts
            V0 = dev(want[0])
            x = few.solve(Sw, Sd, V_init=V0, rule=rule)
            y = one.solve(Sw, Sd, V_init=V0, rule=rule)
            for p, q in zip(x, y):
                assert np.array_equal(p.cpu().numpy(), q.cpu().numpy()), (B, rows, rule)
            assert few.device_status() == 0
            # the profile is of these passes
            few.solve(Sw, Sd, rule=rule, max_iter=20, profile=True)
            torch.cuda.synchronize()
            ms, active = few.last_profile()
            counts = want[1].astype(int)
            assert len(ms) == len(active) == 20 * -(-B // rows) and (ms >= 0).all()
            for p in range(-(-B // rows)):
                mine = counts[p * rows:(p + 1) * rows]
                assert list(active[20 * p:20 * p + 20]) == [(mine > k).sum() for k in range(20)]
            few.close()
            one.close()
    _, word = zbus.zbus_checked_status()
    assert word == 0, hex(word)
    print("passes ok")


if __name__ == "__main__":
    main()
