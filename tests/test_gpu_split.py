"""The plain method's contraction on the tensor cores (csrc/split.cu), from 97
padded unknowns: its edges against the oracle, one map and one adjoint sweep
against extended precision, and its bits against the allocation-free solve,
which runs the batch in other passes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import zbus_oracle as O                      # noqa: E402
from paper_2605_14103_gb300 import feeders as F          # noqa: E402
from paper_2605_14103_gb300 import zbus                  # noqa: E402

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_14103_gb300 import build as B
    B.build()
    zbus.lib()


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


# 99: the smallest size of the path; 192 | 195 and 255 | 258: its N-tiles;
# 384 | 387: whole 64-deep steps and a remainder; 1035: more products per pair
# of digits than one accumulator sums; 2049: eight 256-output tiles and one row
@pytest.mark.parametrize("N,B", [(34, 1), (65, 127), (66, 128), (86, 129), (87, 300), (129, 33),
                                 (130, 2), (346, 7), (684, 3)])
def test_one_map_and_one_adjoint_sweep(N, B):
    """v = w + Z i(w) and mu = Z^T conj(G) within n eps of the largest products
    (the rounding bound of an FP64 sum of n terms, its sqrt(n) in practice)."""
    f = F.make_feeder(N, 1000 + N, delta_frac=0.4)
    Sw, Sd = F.make_scenarios(f, B, 0.5, 1.5)
    net = zbus.Network.from_feeder(f)
    Z, w = (x.cpu().numpy() for x in net.get_z())
    V0 = np.broadcast_to(w, (B, f.n)).copy()
    cur = O.load_currents(V0, Sw, Sd)
    V, it, cv = net.solve(dev(Sw), dev(Sd), max_iter=1)
    ref = (cur.astype(np.clongdouble) @ Z.T.astype(np.clongdouble) + w).astype(np.complex128)
    bound = 4 * EPS + f.n * EPS * np.abs(Z).max() * np.abs(cur).max()
    assert np.abs(V.cpu().numpy() - ref).max() <= bound
    assert (it.cpu().numpy() == 1).all()
    rng = np.random.default_rng(N)
    G = rng.normal(size=Sw.shape) + 1j * rng.normal(size=Sw.shape)
    dw, _, it, _ = net.solve_adjoint(dev(V0), dev(G), None, None, tol=0.0, max_iter=1,
                                     delta=False)
    mu = (np.conj(G).astype(np.clongdouble) @ Z.astype(np.clongdouble)).astype(np.complex128)
    bound = f.n * EPS * np.abs(Z).max() * np.abs(G).max()
    assert np.abs(dw.cpu().numpy() + mu / np.conj(V0)).max() <= bound
    net.close()


@pytest.mark.parametrize("N,B,rule", [(34, 129, "maxabs"), (87, 1, "summag"), (130, 257, "summag"),
                                      (346, 40, "maxabs")])
def test_solve_at_the_edges(N, B, rule):
    f = F.make_feeder(N, 2000 + N, delta_frac=0.4, mult_hi=1.5)
    Sw, Sd = F.make_scenarios(f, B, 0.5, 1.5)
    if B > 2:
        Sw[1] *= 500.0      # far beyond what the feeder carries
        Sd[1] *= 500.0
        Sw[2, 0] = np.inf   # not a number from the first current on
        Sw[0] = Sd[0] = 0   # no load at all: one map
    ok = np.ones(B, dtype=bool)
    ok[1:3] = B <= 2
    ref = O.solve_coo(f.n_total, f.Y_row, f.Y_col, f.Y_val, f.slack_idx, f.v_slack, Sw[ok],
                      Sd[ok], tol=1e-9, rule=rule)
    net = zbus.Network.from_feeder(f)
    V, it, cv = net.solve(dev(Sw), dev(Sd), tol=1e-9, rule=rule)
    assert net.device_status() == 0
    V, it, cv = V.cpu().numpy(), it.cpu().numpy(), cv.cpu().numpy()
    assert np.array_equal(it[ok], ref["iters"]) and np.array_equal(cv[ok], ref["converged"])
    assert np.abs(V[ok] - ref["V"]).max() <= 1e-10
    if B > 2:
        assert it[2] == 1 and cv[2] == 0
        out = torch.empty((B, f.n), dtype=torch.complex128, device="cuda")
        it2 = torch.empty(B, dtype=torch.int32, device="cuda")
        cv2 = torch.empty(B, dtype=torch.uint8, device="cuda")
        zbus.zbus_solve_noalloc(net.handle, dev(Sw), dev(Sd), None, 1e-9, 50, rule, out, it2, cv2)
        assert np.array_equal(out.cpu().numpy()[ok], V[ok])
        assert np.array_equal(it2.cpu().numpy(), it) and np.array_equal(cv2.cpu().numpy(), cv)
    net.close()


def test_a_network_that_ends_inside_a_bus():
    """n not a multiple of 3 (wye loads only)."""
    f = F.make_feeder(80, 77)
    keep = (f.Y_row < f.n_total - 1) & (f.Y_col < f.n_total - 1)
    row, col, val = f.Y_row[keep], f.Y_col[keep], f.Y_val[keep]
    Sw = F.make_scenarios(f, 20, 0.8, 1.2)[0][:, :-1].copy()
    ref = O.solve_coo(f.n_total - 1, row, col, val, f.slack_idx, f.v_slack, Sw, 0 * Sw,
                      bus_phase=np.arange(f.n_total - 1))
    net = zbus.Network(f.n_total - 1, row, col, val, f.slack_idx, f.v_slack)
    V, it, cv = net.solve(dev(Sw))
    assert np.array_equal(it.cpu().numpy(), ref["iters"])
    assert np.array_equal(cv.cpu().numpy(), ref["converged"])
    assert np.abs(V.cpu().numpy() - ref["V"]).max() <= 1e-10
    net.close()
