"""FP32 pair sums on grids so fine that r^2 is no normal FP32 number: the pairs count,
with the kernel's value at r = 0 to FP32 rounding.  Against the oracle with the FP32
path's stated tolerances (E 1e-6, v 1e-5 of max|v|)."""
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


@pytest.mark.parametrize("h", [1e-16, 1e-18, 1e-19, 1e-20, 1e-22, 1e-24])
@pytest.mark.parametrize("dims", [(5, 4, 4), (9, 8, 7)])
@pytest.mark.parametrize("skew", [False, True])
@pytest.mark.parametrize("periodic,cut", [((False,) * 3, 0.0), ((True, False, True), 2.21)])
def test_uniform_density(V, oracle_mod, gtable, oracle_spline, h, dims, skew, periodic, cut):
    """80 and 504 points (ragged, diagonal and whole tiles) of one density, in open cells
    and with images under a cutoff of `cut` spacings."""
    import torch
    r_cut = cut * h
    n = np.full(dims, 0.03)
    cell = np.diag([h * d for d in dims])
    if skew:
        cell[1, 0] = 0.3 * cell[0, 0]
    geo = cell if skew else np.diag(cell)
    # (the gradient is given to the oracle: its stencil's rounding is 1e-17 / h)
    P = oracle_mod.Problem(n, np.diag(cell), periodic, 1e-6, r_cut, oracle_spline, cell=cell if skew else None,
                           g=np.zeros((3,) + dims))
    e = P.energy()
    v = P.potential(e["A"], e["U"])
    t = torch.from_numpy(n).to("cuda:0")
    E, r = V.energy(t, geo, periodic, 1e-6, r_cut, gtable, "fp32")
    Ev, vg, rv = V.potential(t, geo, periodic, 1e-6, r_cut, gtable, "fp32")
    for res in (r, rv):
        assert res["n_active"] == n.size and res["pairs"] == e["pairs"]
    assert abs(E - e["E"]) <= 1e-6 * abs(e["E"])
    assert abs(Ev - e["E"]) <= 1e-6 * abs(e["E"])
    assert np.max(np.abs(vg.cpu().numpy() - v)) <= 1e-5 * np.max(np.abs(v))
