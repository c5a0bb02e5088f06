"""FP64 pairs so far past the table that eq. (17)'s denominator, about 27 (q r)^7 with
D, leaves the range of FP64: they contribute nothing, and the call succeeds.  Against
the oracle with the FP64 path's stated tolerance (1e-10)."""
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


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to("cuda:0")


DIMS, L = (9, 8, 10), (6.0, 5.6, 7.0)


@pytest.mark.parametrize("q", [1e12, 1e20, 1e21, 1e30, 1e42, 1e43, 3e43, 1e44, 1e45, 1e60, 1e100])
@pytest.mark.parametrize("periodic,r_cut", [((False,) * 3, 0.0), ((True, True, False), 6.5)])
def test_energy_with_a_given_gradient(V, oracle_mod, gtable, oracle_spline, q, periodic, r_cut):
    """One point whose gradient makes its q0 about q."""
    rng = np.random.default_rng(3)
    n = 0.05 * np.exp(0.3 * rng.uniform(-1, 1, DIMS))
    g = 0.02 * rng.normal(size=(3,) + DIMS)
    kF = (3.0 * np.pi ** 2 * n[4, 4, 4]) ** (1.0 / 3.0)
    g[:, 4, 4, 4] = (n[4, 4, 4] * np.sqrt(q * 36.0 / 0.8491 * kF), 0.0, 0.0)
    P = oracle_mod.Problem(n, L, periodic, 1e-6, r_cut, oracle_spline, g=g)
    assert 0.9 * q <= P.qa.max() <= 1.1 * q
    e = P.energy()
    E, r = V.energy(_t(n), L, periodic, 1e-6, r_cut, gtable, "fp64", grad=_t(g))
    assert r["pairs"] == e["pairs"]
    assert abs(E - e["E"]) <= 1e-10 * abs(e["E"])


@pytest.mark.parametrize("low", [1e-12, 1e-20, 1e-21, 1e-24, 1e-30])
def test_potential_beside_a_steep_density(V, oracle_mod, gtable, oracle_spline, low):
    """Points of density `low` beside ordinary ones (q0 up to about 1 / low^(7/3)), all above the cutoff."""
    rng = np.random.default_rng(4)
    n = np.full(DIMS, low)
    n[2:6, 2:6, 2:6] = 0.05 * np.exp(0.3 * rng.uniform(-1, 1, (4, 4, 4)))
    P = oracle_mod.Problem(n, L, (False,) * 3, 0.1 * low, 0.0, oracle_spline)
    e = P.energy()
    v = P.potential(e["A"], e["U"])
    E, vg, r = V.potential(_t(n), L, (False,) * 3, 0.1 * low, 0.0, gtable, "fp64")
    assert r["pairs"] == e["pairs"] and r["n_active"] == n.size
    assert abs(E - e["E"]) <= 1e-10 * abs(e["E"])
    assert np.max(np.abs(vg.cpu().numpy() - v)) <= 1e-10 * np.max(np.abs(v))
