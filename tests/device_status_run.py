"""Child process of tests/test_gpu_giveup_f64.py, in the checked build: what
zbus_last_device_status reports belongs to the last solve of that network,
whatever happened to the scratch or to other networks since.  Prints
"status ok" on success."""
import os
import sys

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from paper_2605_14103_gb300 import feeders as F          # noqa: E402
from paper_2605_14103_gb300 import zbus                  # noqa: E402

ZBUS_ERR_TIMEOUT = 5


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def noalloc(net, Sw, Sd):
    B, n = Sw.shape
    zbus.zbus_solve_noalloc(net.handle, dev(Sw), dev(Sd), None, 1e-8, 50, "maxabs",
                            torch.empty((B, n), dtype=torch.complex128, device="cuda"),
                            torch.empty(B, dtype=torch.int32, device="cuda"),
                            torch.empty(B, dtype=torch.uint8, device="cuda"))


def gives_up(call):
    zbus._check(zbus.lib().zbus_checked_set_wait(0))
    try:
        call()
        torch.cuda.synchronize()
    finally:
        zbus._check(zbus.lib().zbus_checked_set_wait(2000000000))


def main():
    flag, _ = zbus.zbus_checked_status()
    assert flag == 1, "not the checked build"
    f = F.make_feeder(60, 1, delta_frac=0.3)
    Sw, Sd = F.make_scenarios(f, 40, 0.8, 1.2)
    a, b = zbus.Network.from_feeder(f), zbus.Network.from_feeder(f)
    # the scratch has grown since
    a.solve(dev(Sw), dev(Sd))
    zbus.zbus_network_reserve(a.handle, 5000, "fp64")
    assert a.device_status() == 0
    gives_up(lambda: a.solve(dev(Sw), dev(Sd)))
    zbus.zbus_network_reserve(a.handle, 20000, "fp64")
    assert a.device_status() == ZBUS_ERR_TIMEOUT
    # another network's allocation-free solve came after
    gives_up(lambda: noalloc(a, Sw, Sd))
    noalloc(b, Sw, Sd)
    assert a.device_status() == ZBUS_ERR_TIMEOUT and b.device_status() == 0
    gives_up(lambda: noalloc(b, Sw, Sd))
    noalloc(a, Sw, Sd)
    assert a.device_status() == 0 and b.device_status() == ZBUS_ERR_TIMEOUT
    # a mixed batch whose group is gone since (its other network closed)
    gives_up(lambda: a.solve(dev(Sw), dev(Sd)))
    zbus.solve_batched([a, b], [(dev(Sw), dev(Sd))] * 2, precision="fp16_scaled")
    assert a.device_status() == 0 and b.device_status() == 0
    b.close()
    assert a.device_status() == 0
    a.close()
    print("status ok")


if __name__ == "__main__":
    main()
