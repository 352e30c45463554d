"""Child process of tests/test_gpu_giveup_f64.py, in the checked build: the
plain FP64 form's contraction (csrc/split.cu) gives up its waits (limit 0), in
the solve, the dense gradient and the allocation-free solve; the failure is
reported, no scenario is flagged as converged, and the next ordinary call is
right.  Prints "giveup ok" on success."""
import os
import sys

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from oracle import zbus_oracle as O                      # noqa: E402
from paper_2605_14103_gb300 import feeders as F          # noqa: E402
from paper_2605_14103_gb300 import zbus                  # noqa: E402

ZBUS_ERR_TIMEOUT = 5


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def main():
    flag, word = zbus.zbus_checked_status()
    assert flag == 1, "not the checked build"
    B = 300
    for N in (34, 130):        # two widths of the contraction's tile
        f = F.make_feeder(N, 202, delta_frac=0.3)
        Sw, Sd = F.make_scenarios(f, B, 0.8, 1.2, seed=9)
        G = np.random.default_rng(N).normal(size=Sw.shape) * (1 - 0.5j)
        r = O.solve_coo(f.n_total, f.Y_row, f.Y_col, f.Y_val, f.slack_idx, f.v_slack, Sw, Sd)
        rv = O.solve_coo(f.n_total, f.Y_row, f.Y_col, f.Y_val, f.slack_idx, f.v_slack, Sw, Sd,
                         tol=1e-14, max_iter=300)
        Hw, Hd = O.solve_adjoint(rv["Z"], rv["V"], Sw, Sd, G)
        net = zbus.Network.from_feeder(f)

        def solve():
            V, it, cv = net.solve(dev(Sw), dev(Sd))
            return np.abs(V.cpu().numpy() - r["V"]).max() <= 1e-9, cv

        def gradient():
            dw, dd, it, cv = net.solve_adjoint(dev(rv["V"]), dev(G), dev(Sw), dev(Sd))
            return (np.abs(dw.cpu().numpy() - Hw).max() <= 1e-9 * np.abs(Hw).max() and
                    np.abs(dd.cpu().numpy() - Hd).max() <= 1e-9 * np.abs(Hd).max()), cv

        def noalloc():
            V = torch.empty((B, f.n), dtype=torch.complex128, device="cuda")
            it = torch.empty(B, dtype=torch.int32, device="cuda")
            cv = torch.empty(B, dtype=torch.uint8, device="cuda")
            zbus.zbus_solve_noalloc(net.handle, dev(Sw), dev(Sd), None, 1e-8, 50, "maxabs", V, it,
                                    cv)
            return np.abs(V.cpu().numpy() - r["V"]).max() <= 1e-9, cv

        for call in (solve, gradient, noalloc):
            for limit in (2000000000, 0, 2000000000):
                zbus._check(zbus.lib().zbus_checked_set_wait(limit))
                try:
                    right, cv = call()
                    st = net.device_status()
                finally:
                    zbus._check(zbus.lib().zbus_checked_set_wait(2000000000))
                if limit:
                    assert st == 0 and right and cv.cpu().numpy().all(), (N, call.__name__, st)
                else:
                    assert st == ZBUS_ERR_TIMEOUT, (N, call.__name__, st)
                    assert not cv.cpu().numpy().any(), (N, call.__name__)
        net.close()
    flag, word = zbus.zbus_checked_status()
    assert word == 0, hex(word)
    print("giveup ok")


if __name__ == "__main__":
    main()
