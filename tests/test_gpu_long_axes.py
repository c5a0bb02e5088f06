"""The FP64 pair sums on axes of more than a million cells, where the table of
distances over index displacements would not hold every displacement: all pairs
count, against the oracle with the FP64 path's stated tolerance (1e-10)."""
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


@pytest.fixture(scope="module")
def gtable(V, oracle_table):
    return V.Table.from_nodes(oracle_table, 30.0)


def _plateaus(dims, at):
    """Five equal points around each index along the longest axis: no gradient at its own
    point, so that q0 is ordinary there however short the spacing is."""
    ax = int(np.argmax(dims))
    n = np.zeros(dims)
    for c in at:
        idx = [slice(None)] * 3
        idx[ax] = [(c + o) % dims[ax] for o in (-2, -1, 0, 1, 2)]
        n[tuple(idx)] = 0.05 + 0.01 * (c % 7)
    return n


CASES = {
    # name: (dims, cell rows, periodic, r_cut, plateau centres); spans of 1,048,573 cells
    # without images, and of 1.2 million cells of a short periodic axis
    "open": ((1048576, 1, 1), np.diag((12.0, 3.0, 3.0)), (False, False, False), 0.0, (2, 500000, 1048573)),
    "open, last axis": ((1, 1, 1048576), np.diag((3.0, 3.0, 12.0)), (False, False, False), 0.0, (2, 1048573)),
    "open, cutoff": ((1048576, 1, 2), np.diag((12.0, 3.0, 3.0)), (False, False, False), 30.0, (2, 1048573)),
    "open, skewed": ((1048576, 1, 1), np.array([[12.0, 0.3, 0.0], [0.0, 3.0, 0.0], [0.1, 0.0, 3.0]]),
                     (False, False, False), 0.0, (2, 1048573)),
    "periodic": ((40000, 1, 1), np.diag((0.5, 3.0, 3.0)), (True, False, False), 15.0, (7, 20000)),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_every_pair_counts(V, oracle_mod, gtable, oracle_spline, name):
    import torch
    dims, cell, periodic, r_cut, at = CASES[name]
    n = _plateaus(dims, at)
    diagonal = np.array_equal(cell, np.diag(np.diag(cell)))
    P = oracle_mod.Problem(n, np.diag(cell), periodic, 1e-6, r_cut, oracle_spline, cell=None if diagonal else cell)
    e = P.energy()
    t = torch.from_numpy(n).to("cuda:0")
    geo = np.diag(cell) if diagonal else cell
    E, r = V.energy(t, geo, periodic, 1e-6, r_cut, gtable, "fp64")
    Ev, v, rv = V.potential(t, geo, periodic, 1e-6, r_cut, gtable, "fp64")
    for res in (r, rv):
        assert res["n_active"] == P.n_active and res["pairs"] == e["pairs"]
    assert abs(E - e["E"]) <= 1e-10 * abs(e["E"])
    assert abs(Ev - e["E"]) <= 1e-10 * abs(e["E"])
    # E without the self terms, which are most of it
    x = e["E"] - e["E_diag"]
    assert abs((E - r["E_diag"]) - x) <= 1e-10 * abs(e["E"])
