"""The plain method's contraction on the tensor cores (csrc/split.cu) where the
entries of a row differ in size: every row's error is bounded by its own terms,
as an FP64 sum's is, not by the largest entry of the operand."""
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


def magnitude(x):
    return np.abs(x.real) + np.abs(x.imag)


# sizes of the other entries against one bus (or a twentieth of the entries)
# of size one, or spread over twelve decades
SPREADS = [1e-2, 1e-4, 1e-8, 1e-12, 0.0, "log"]


def spread(x, how, at, rng):
    """x [B][n] with entries of sizes `how` apart; row b keeps those of bus at[b]."""
    if how == "log":
        return x * 10.0 ** rng.uniform(-12, 0, size=x.shape)
    s = np.full(x.shape, how)
    for b, a in enumerate(at):
        s[b, 3 * a:3 * a + 3] = 1.0
    return x * s


@pytest.mark.parametrize("how", SPREADS, ids=str)
@pytest.mark.parametrize("N", [34, 87, 301])
def test_rows_of_entries_of_different_size(N, how):
    """One map and one adjoint sweep: |error_i| <= 4 sqrt(n) eps S_i, S_i the
    sum of the row's |Re| + |Im| products (an FP64 sum of n rounded products,
    errors independent: sqrt(n) eps S_i and less), and the rounding of v."""
    f = F.make_feeder(N, 3000 + N)
    n, B = f.n, 12
    rng = np.random.default_rng(N)
    net = zbus.Network.from_feeder(f)
    Z, w = (x.cpu().numpy() for x in net.get_z())
    kids = [k - 1 for k in range(1, N) if f.parent[k] == 0]   # buses at the slack
    at = (kids + list(rng.permutation(N - 1)))[:B]
    Sw = spread(F.make_scenarios(f, B, 0.5, 1.5)[0], how, at, rng)
    V0 = np.broadcast_to(w, (B, n)).copy()
    V, _, _ = net.solve(dev(Sw), None, max_iter=1)
    cur = O.load_currents(V0, Sw, 0 * Sw)
    ref = cur.astype(np.clongdouble) @ Z.T.astype(np.clongdouble) + w
    S = magnitude(cur) @ magnitude(Z).T
    err = np.abs((V.cpu().numpy() - ref).astype(np.complex128))
    assert (err <= 4 * np.sqrt(n) * EPS * S + 2 * EPS * np.abs(ref).astype(float)).all()
    G = spread(rng.normal(size=Sw.shape) + 1j * rng.normal(size=Sw.shape), how, at, rng)
    dw, _, _, _ = net.solve_adjoint(dev(V0), dev(G), None, None, tol=0.0, max_iter=1,
                                    delta=False)
    mu = np.conj(G).astype(np.clongdouble) @ Z.astype(np.clongdouble)
    S = magnitude(G) @ magnitude(Z)
    err = np.abs((dw.cpu().numpy() * np.conj(V0) + mu).astype(np.complex128))
    # dw = -mu / conj(V): the quotient and its product here round eight times
    assert (err <= (4 * np.sqrt(n) + 8) * EPS * S).all()
    net.close()


@pytest.mark.parametrize("N", [34, 346])
def test_each_scenario_alone_and_in_the_batch(N):
    """Scenarios of every spread, one without loads, one of an infinite load:
    the same bits alone as in one batch."""
    f = F.make_feeder(N, 4000 + N, delta_frac=0.3)
    rng = np.random.default_rng(N)
    Sw, Sd = F.make_scenarios(f, 2 * len(SPREADS) + 2, 0.5, 1.2)
    for k, how in enumerate(2 * SPREADS):
        at = [int(rng.integers(N - 1))]
        Sw[k] = spread(Sw[k][None], how, at, rng)[0]
        Sd[k] = spread(Sd[k][None], how, at, rng)[0]
    Sw[-2] = Sd[-2] = 0
    Sw[-1, 0] = np.inf
    net = zbus.Network.from_feeder(f)
    V, it, cv = (x.cpu().numpy() for x in net.solve(dev(Sw), dev(Sd)))
    ok = O.solve_coo(f.n_total, f.Y_row, f.Y_col, f.Y_val, f.slack_idx, f.v_slack, Sw[:-1],
                     Sd[:-1])
    assert np.abs(V[:-1] - ok["V"]).max() <= 1e-10 and cv[:-1].all() and not cv[-1]
    assert it[-2] == 1 and it[-1] == 1
    for b in range(len(Sw)):
        Va, ia, ca = (x.cpu().numpy() for x in net.solve(dev(Sw[b:b + 1]), dev(Sd[b:b + 1])))
        assert np.array_equal(Va[0], V[b], equal_nan=True) and ia[0] == it[b] and ca[0] == cv[b]
    net.close()
