"""The count of pairs past the last delta node (n_clamped) against the oracle, exactly,
in both precisions and both modes: ragged and whole tiles, pairs partly inside a
cutoff, images, skewed and open cells.  Few delta nodes and densities with steep
places, so that a good part of the pairs is counted; no pair's delta is near enough to
the last node for FP32 to tell otherwise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import __graft_entry__
    __graft_entry__.build()
    import paper_0810_2273_gb300 as V
    return V


NODES = (30, 6)
SEED = 3000
CELLS = {
    "open": (np.diag((5.0, 4.4, 4.0)), (False, False, False), 0.0),
    "open, cutoff": (np.diag((5.0, 4.4, 4.0)), (False, False, False), 3.7),
    "slab": (np.diag((5.0, 4.4, 8.0)), (True, True, False), 6.5),
    "skew": (np.array([[5.0, 0.0, 0.0], [1.9, 4.2, 0.0], [0.7, -0.4, 6.0]]), (True, False, True), 6.0),
    "skew, open": (np.array([[5.0, 0.0, 0.0], [1.9, 4.2, 0.0], [0.7, -0.4, 6.0]]), (False, False, False), 0.0),
}


def nodes():
    D = np.linspace(0.0, 12.0, NODES[0])[:, None]
    dl = (np.arange(NODES[1]) / NODES[1])[None, :]
    return (1.0 - 0.3 * dl ** 2) * np.exp(-0.2 * D) * np.cos(0.3 * D) - 1e-3


def density(dims, active):
    """The first `active` points, neighbours that differ by up to a factor of a thousand
    (q0 spans two to five decades), and nothing elsewhere."""
    n = np.zeros(dims)
    n.ravel()[:active] = 0.05 * 10.0 ** np.random.default_rng(SEED + active).uniform(-1.5, 1.5, active)
    return n


def problem(oracle_mod, kind, active):
    cell, periodic, r_cut = CELLS[kind]
    n = density((9, 8, 7), active)
    n_cut = 1e-6
    diagonal = np.array_equal(cell, np.diag(np.diag(cell)))
    P = oracle_mod.Problem(n, np.diag(cell), periodic, n_cut, r_cut, oracle_mod.Spline(nodes(), 12.0),
                           cell=None if diagonal else cell)
    return P, np.diag(cell) if diagonal else cell


@pytest.mark.parametrize("kind", sorted(CELLS))
@pytest.mark.parametrize("active", [33, 64, 97, 129, 321, 504])
def test_clamp_counts(V, oracle_mod, kind, active):
    import torch
    P, geo = problem(oracle_mod, kind, active)
    q = P.qa
    dl = np.abs(q[:, None] - q[None, :]) / (q[:, None] + q[None, :]) * NODES[1]
    assert np.min(np.abs(dl - (NODES[1] - 1))) > 1e-5
    e = P.energy()
    assert 0 < e["clamped"] < e["pairs"]
    table = V.Table.from_nodes(nodes(), 12.0)
    t = torch.from_numpy(P.n).to("cuda:0")
    for precision in ("fp32", "fp64"):
        _, r = V.energy(t, geo, P.periodic, P.n_cut, P.rc, table, precision)
        _, _, rv = V.potential(t, geo, P.periodic, P.n_cut, P.rc, table, precision)
        for res in (r, rv):
            assert (res["pairs"], res["n_clamped"]) == (e["pairs"], e["clamped"]), precision
