"""Newton-Raphson on grids that reach the edges of the preconditioner's
layout: tiles of 32 rows, levels just within and beyond the 128 rows that one
warp takes, its steps of up to 32 rows, and Gram-Schmidt beyond one chunk of
eight vectors."""
import numpy as np
import pytest
import torch

from oracle import nr_oracle as O
from paper_2605_14103_gb300 import zbus

pytestmark = pytest.mark.gpu


def network(N, kind, seed):
    """COO of a chain, a star, a star of chains, or lines side by side at the
    slack; every third bus PV."""
    if kind == "chain":
        edges = [(k - 1, k) for k in range(1, N)]
    elif kind == "star":
        edges = [(0, k) for k in range(1, N)]
    elif kind == "hub":          # a PQ hub with chains of two
        edges = [(0, 1)] + [(1 if k % 2 == 0 else k - 1, k) for k in range(2, N)]
    else:                        # a ladder: two chains with rungs
        edges = [(max(k - 2, 0), k) for k in range(1, N)] + [(k, k + 1) for k in range(1, N - 1, 2)]
        edges = sorted(set((min(e), max(e)) for e in edges))
    rng = np.random.default_rng(seed)
    x = rng.uniform(0.5, 1.5, len(edges)) * 0.2 / N
    y = 1.0 / (0.2 * x + 1j * x)
    row, col, val = [], [], []
    for (a, b), v in zip(edges, y):
        row += [a, b, a, b]
        col += [a, b, b, a]
        val += [v, v, -v, -v]
    bt = np.where(np.arange(N) % 3 == 2, 1, 0).astype(np.int32)
    bt[0] = 2
    return row, col, np.array(val), bt, np.where(bt == 0, 1.0, 1.01)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", ["chain", "star", "hub", "ladder"])
@pytest.mark.parametrize("N", [2, 5, 33, 65, 129, 130, 161])
def test_layout_edges_against_the_oracle(N, kind, prec):
    row, col, val, bt, vs = network(N, kind, N)
    rng = np.random.default_rng(3)
    P, Q = rng.uniform(-0.5, 0.2, (3, N)), rng.uniform(-0.2, 0.1, (3, N))
    ref = O.solve_batch(N, row, col, val, bt, vs, P, Q)
    assert ref["converged"].all()
    net = zbus.NrNetwork(N, row, col, val, bt, vs)
    d = [torch.from_numpy(a).cuda() for a in (P, Q)]
    # the second call needs more than eight Krylov vectors wherever there are as many unknowns
    for tol in (1e-6, 1e-13 if prec == "fp64" else 1e-6):
        V, it, cv, gm = net.solve(*d, precision=prec, gmres_tol=tol)
        np.testing.assert_array_equal(cv.cpu().numpy(), ref["converged"])
        assert np.abs(V.cpu().numpy() - ref["V"]).max() <= 1e-8
        assert np.abs(it.cpu().numpy() - ref["iters"]).max() <= 1
    net.close()
