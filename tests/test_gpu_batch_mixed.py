"""Orthogonal cells of a batch run as skewed cells only in a launch (24 instances) that
holds a skewed one: the others run as they would without it."""
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


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-6), ("fp64", 1e-12)])
@pytest.mark.parametrize("where", [0, 5, 24, 29])
def test_skewed_cell_in_one_of_two_launches(V, oracle_table, precision, tol, where):
    import torch
    table = V.Table.from_nodes(oracle_table, 30.0)
    rng = np.random.default_rng(where)
    orth, skew = (5.0, 4.4, 6.0), np.array([[5.0, 0.0, 0.0], [1.9, 4.2, 0.0], [0.7, -0.4, 6.0]])
    ns = [torch.from_numpy(0.05 * np.exp(0.3 * rng.uniform(-1, 1, (7 + k % 3, 8, 7)))).to("cuda:0") for k in range(30)]
    geo = [skew if k == where else orth for k in range(30)]
    per = [(True, True, False)] * 30
    E, r = V.energy_batched(ns, geo, per, 1e-6, 6.0, table, precision)
    for k in range(30):
        one, _ = V.energy(ns[k], geo[k], per[k], 1e-6, 6.0, table, precision)
        assert abs(E[k] - one) <= tol * abs(one)
    # launches: those of the two halves by themselves (Cartesian boxes only where a skewed cell is)
    parts = [V.energy_batched(ns[a:b], geo[a:b], per[a:b], 1e-6, 6.0, table, precision)[1]["launches"]
             for a, b in ((0, 24), (24, 30))]
    assert r["launches"] == sum(parts)
    table.free()
