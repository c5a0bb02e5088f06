"""Skewed cells whose points lie thousands of cutoffs from the origin: the boxes that
select images are Cartesian FP32 numbers there, and their rounding must neither drop a
pair just inside the cutoff nor admit one just outside.  Pair counts exact."""
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


@pytest.mark.parametrize("side", [-1.0, 1.0])
@pytest.mark.parametrize("disp", [(4, 3, 3), (7, 3, 5), (8, 0, 0), (3, 7, 2)])
@pytest.mark.parametrize("start", [59977, 41003])
def test_pairs_at_the_cutoff(V, oracle_mod, gtable, oracle_spline, side, disp, start):
    """20 x 8 x 8 points at the far end of a 42,000 bohr axis; the cutoff 2e-5 beside the
    distance of a displacement, so that many pairs lie just inside or just outside."""
    import torch
    dims = (60000, 8, 8)
    v = np.array([[0.7, 0.0, 0.0], [0.0, 0.61, 0.0], [0.0, 1e-3, 0.53]])
    cell = v * np.array(dims, dtype=float)[:, None]
    rng = np.random.default_rng(9)
    n = np.zeros(dims)
    n[start:start + 20] = 0.05 * np.exp(0.2 * rng.uniform(-1, 1, (20, 8, 8)))
    r_cut = float(np.linalg.norm(np.array(disp) @ v)) * (1.0 + side * 2e-5)
    P = oracle_mod.Problem(n, None, (False,) * 3, 1e-6, r_cut, oracle_spline, cell=cell)
    e = P.energy()
    t = torch.from_numpy(n).to("cuda:0")
    for precision, tol in (("fp32", 1e-6), ("fp64", 1e-10)):
        E, r = V.energy(t, cell, (False,) * 3, 1e-6, r_cut, gtable, precision)
        Ev, _, rv = V.potential(t, cell, (False,) * 3, 1e-6, r_cut, gtable, precision)
        assert (r["pairs"], rv["pairs"]) == (e["pairs"], e["pairs"]), precision
        assert abs(E - e["E"]) <= tol * abs(e["E"]) and abs(Ev - e["E"]) <= tol * abs(e["E"])
