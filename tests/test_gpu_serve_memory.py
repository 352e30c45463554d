"""The serving loop's device memory beside what the plain FP64 form keeps of its
networks: the slices of Z and the scratch of its sweeps."""
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


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def pool_and_budget(room):
    """Two networks that hold their mixed operands, requests for both, and a
    budget of 128 slots and every operand with `room` bytes left."""
    feeders = [F.make_feeder(N, 50 + N, delta_frac=0.3) for N in (40, 100)]
    nets = [zbus.Network.from_feeder(f) for f in feeders]
    loads = [[dev(x) for x in F.make_scenarios(f, 60, 0.8, 1.2)] for f in feeders]
    reqs = [{"feeder": k, "S_wye": sw, "S_delta": sd} for k, (sw, sd) in enumerate(loads)]
    zbus.serve(nets, reqs, max_slots=128)
    foot = [zbus.zbus_serve_footprint(net.handle, "fp16_scaled") for net in nets]
    budget = sum(o + 128 * s for o, _, s in foot) + max(x for _, x, _ in foot) + room
    return feeders, nets, loads, reqs, budget


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def slices(f):
    return 22 * f.n * ((f.n + 63) // 64 * 64) * 2 + 8 * f.n


def test_sweep_scratch_outside_the_budget_is_given_back():
    # room for the slices of both and not for the scratch of 8192 scenarios
    feeders, nets, loads, reqs, budget = pool_and_budget(2 << 20)
    budget += sum(slices(f) for f in feeders)
    assert sum(slices(f) for f in feeders) < 16 << 20
    for net in nets:
        zbus.zbus_network_reserve(net.handle, 8192, "fp64")
    scratch = sum(8192 * 22 * 6 * f.n for f in feeders)     # its planes alone
    zbus.serve(nets, reqs, max_slots=128)       # workspaces of this size: no budget reached
    before = free_bytes()
    zbus.serve(nets, reqs, max_slots=128, hbm_budget_bytes=budget)
    assert free_bytes() - before >= scratch - (64 << 20)
    # the next solve takes it again
    for f, net, (sw, sd) in zip(feeders, nets, loads):
        V, it, cv = net.solve(sw, sd)
        assert cv.cpu().numpy().all()
        net.close()


@pytest.mark.parametrize("evict", [False, True])
def test_allocation_free_solve_after_a_tight_serving_loop(evict):
    """The same bits as zbus_solve, whether the loop gave up only the slices
    (no room beside the cache) or a network's operands in turn with the
    other's, and formed them again."""
    feeders, nets, loads, reqs, budget = pool_and_budget(1 << 20)
    if evict:   # the cache holds the larger network's operands alone
        budget -= zbus.zbus_serve_footprint(nets[0].handle, "fp16_scaled")[0] // 2
    for _ in range(2):
        zbus.serve(nets, reqs, max_slots=128, hbm_budget_bytes=budget)
        for f, net, (sw, sd) in zip(feeders, nets, loads):
            B = sw.shape[0]
            out = torch.empty((B, f.n), dtype=torch.complex128, device="cuda")
            it = torch.empty(B, dtype=torch.int32, device="cuda")
            cv = torch.empty(B, dtype=torch.uint8, device="cuda")
            try:
                zbus.zbus_solve_noalloc(net.handle, sw, sd, None, 1e-8, 50, "maxabs", out, it, cv)
            except zbus.ZbusError as e:    # evicted at the end: refused, not answered otherwise
                assert evict and "zbus_network_reserve" in str(e)
                continue
            V, it2, cv2 = net.solve(sw, sd)
            assert np.array_equal(out.cpu().numpy(), V.cpu().numpy())
            assert np.array_equal(it.cpu().numpy(), it2.cpu().numpy())
            assert np.array_equal(cv.cpu().numpy(), cv2.cpu().numpy())
    for net in nets:
        net.close()
