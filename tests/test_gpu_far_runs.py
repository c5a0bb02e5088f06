"""The far tail's sums where their parts change: a q0 range so wide that a run of
doubling nodes takes more than one block column, planes too many for the shared
tables, and three periodic axes (one plane split over blocks).  Against the oracle's
plain O(N^2) sum with the bars of the far-tail parity tests: T 1e-11, v 1e-10 of its
largest value."""
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


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to("cuda:0")


def _sharp(dims, L, a=0.25):
    """One steep atom: q0 grows without bound into its tail."""
    x = np.meshgrid(*[(np.arange(d) + 0.3) / d * l for d, l in zip(dims, L)], indexing="ij")
    r = np.sqrt(sum((c - 0.47 * l) ** 2 for c, l in zip(x, L)))
    return 3.0 * np.exp(-r / a)


CASES = {
    # name: (dims, lengths, periodic, n_cut, at least this many nodes)
    "wide, planes": ((9, 8, 16), (4.0, 4.2, 14.0), (True, True, False), 1e-22, 230),
    "wide, three axes": ((9, 8, 16), (4.0, 4.2, 14.0), (True, True, True), 1e-22, 230),
    "wide, lines": ((6, 13, 12), (3.0, 11.0, 12.0), (True, False, False), 1e-20, 230),
    "many planes": ((3100, 4, 3), (400.0, 4.0, 4.2), (False, True, True), 1e-25, 1),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_far_tail_parts(V, oracle_mod, oracle_spline, name):
    dims, L, periodic, n_cut, least = CASES[name]
    n = _sharp(dims, L, 0.25 if name != "many planes" else 0.8)
    P = oracle_mod.Problem(n, L, periodic, n_cut, 9.0, oracle_spline)
    T = P.far_tail()
    v = P.far_tail_potential()
    r, vg = V.far_tail(_t(n), L, periodic, n_cut, 9.0, want_v=True)
    assert r["n_active"] == P.n_active and r["nodes"] >= least
    assert abs(r["T"] - T) <= 1e-11 * abs(T)
    # (where the density underflows the oracle's q0 has no derivative and v is NaN)
    ok = np.isfinite(v)
    assert ok.sum() >= P.n_active
    assert np.max(np.abs(vg.cpu().numpy() - v)[ok]) <= 1e-10 * np.max(np.abs(v[ok]))
