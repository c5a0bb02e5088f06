"""The FP32 pair kernel at the sizes where its tiles can go wrong: numbers of active
points around multiples of 32 and 64 (one warp's j and i points), few shared table
rows, and tables without a texture copy (an axis beyond the device's limit for
texture gathers).  Against the FP64 oracle with the FP32 path's stated tolerances: E
1e-6 relative, v 1e-5 of max|v|, pair and clamp counts exact."""
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


# cells: open, a slab whose images cross a short cutoff, and a skewed one
CELLS = {
    "open": (np.diag((5.0, 4.4, 4.0)), (False, False, False), 0.0),
    "slab": (np.diag((5.0, 4.4, 8.0)), (True, True, False), 6.5),
    "skew": (np.array([[5.0, 0.0, 0.0], [1.9, 4.2, 0.0], [0.7, -0.4, 6.0]]), (True, False, True), 6.0),
}


def _density(dims, cell, seed):
    """A smooth positive density with a different value at every point."""
    rng = np.random.default_rng(seed)
    u = np.meshgrid(*[np.arange(d) / d for d in dims], indexing="ij")
    n = np.zeros(dims)
    for _ in range(4):
        k = rng.integers(-1, 2, 3)
        n += rng.uniform(0.2, 0.6) * np.cos(2 * np.pi * (k[0] * u[0] + k[1] * u[1] + k[2] * u[2] + rng.uniform()))
    return 0.05 * np.exp(n) * (1.0 + 0.01 * rng.uniform(-1, 1, dims))


def _check(V, oracle_mod, table, spline, n, cell, periodic, n_cut, r_cut, tuning=None):
    diagonal = np.array_equal(cell, np.diag(np.diag(cell)))
    P = oracle_mod.Problem(n, np.diag(cell), periodic, n_cut, r_cut, spline, cell=None if diagonal else cell)
    e = P.energy()
    v = P.potential(e["A"], e["U"])
    geo = np.diag(cell) if diagonal else cell
    E, r = V.energy(_t(n), geo, periodic, n_cut, r_cut, table, "fp32", tuning=tuning)
    Ev, vg, rv = V.potential(_t(n), geo, periodic, n_cut, r_cut, table, "fp32", tuning=tuning)
    assert abs(E - e["E"]) <= 1e-6 * abs(e["E"])
    assert abs(Ev - e["E"]) <= 1e-6 * abs(e["E"])
    assert np.max(np.abs(vg.cpu().numpy() - v)) <= 1e-5 * np.max(np.abs(v))
    for res in (r, rv):
        assert res["n_active"] == P.n_active and res["pairs"] == e["pairs"]


@pytest.mark.parametrize("kind", sorted(CELLS))
@pytest.mark.parametrize("active", [1, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 193])
def test_active_counts(V, oracle_mod, gtable, oracle_spline, kind, active):
    cell, periodic, r_cut = CELLS[kind]
    dims = (9, 8, 7)
    n = _density(dims, cell, active)
    s = np.sort(n, axis=None)[::-1]
    n_cut = 0.5 * (s[active - 1] + s[active])
    _check(V, oracle_mod, gtable, oracle_spline, n, cell, periodic, n_cut, r_cut)


@pytest.mark.parametrize("rows", [-1, 1, 3, 4, 5, 40])
@pytest.mark.parametrize("row0", [0, 7, 10000])
def test_few_band_rows(V, oracle_mod, gtable, oracle_spline, rows, row0):
    cell, periodic, r_cut = CELLS["slab"]
    n = _density((9, 8, 7), cell, 5)
    _check(V, oracle_mod, gtable, oracle_spline, n, cell, periodic, 1e-6, r_cut,
           tuning={"smem_rows": rows, "smem_row0": row0})


@pytest.mark.parametrize("shape", [(4, 4), (9, 5), (33000, 4)])
def test_table_shapes(V, oracle_mod, shape):
    """The smallest table, a small one, and one with more rows than a texture takes.
    The nodes are those of a smooth kernel-like function: the spline is what counts."""
    nD, nd = shape
    D = np.linspace(0.0, 12.0, nD)[:, None]
    dl = (np.arange(nd) / nd)[None, :]
    nodes = (1.0 - 0.3 * dl ** 2) * np.exp(-0.2 * D) * np.cos(0.3 * D) - 1e-3
    table = V.Table.from_nodes(nodes, 12.0)
    spline = oracle_mod.Spline(nodes, 12.0)
    cell, periodic, r_cut = CELLS["slab"]
    n = _density((9, 8, 7), cell, 6)
    _check(V, oracle_mod, table, spline, n, cell, periodic, 1e-6, r_cut)


def _check_fp64(V, oracle_mod, table, spline, n, cell, periodic, n_cut, r_cut):
    """The FP64 path against the oracle with its stated tolerances: E and v 1e-10."""
    diagonal = np.array_equal(cell, np.diag(np.diag(cell)))
    P = oracle_mod.Problem(n, np.diag(cell), periodic, n_cut, r_cut, spline, cell=None if diagonal else cell)
    e = P.energy()
    v = P.potential(e["A"], e["U"])
    geo = np.diag(cell) if diagonal else cell
    E, r = V.energy(_t(n), geo, periodic, n_cut, r_cut, table, "fp64")
    Ev, vg, rv = V.potential(_t(n), geo, periodic, n_cut, r_cut, table, "fp64")
    assert abs(E - e["E"]) <= 1e-10 * abs(e["E"])
    assert abs(Ev - e["E"]) <= 1e-10 * abs(e["E"])
    assert np.max(np.abs(vg.cpu().numpy() - v)) <= 1e-10 * np.max(np.abs(v))
    for res in (r, rv):
        assert res["n_active"] == P.n_active and res["pairs"] == e["pairs"]


@pytest.mark.parametrize("kind", sorted(CELLS))
@pytest.mark.parametrize("active", [1, 31, 32, 33, 64, 65, 97])
def test_active_counts_fp64(V, oracle_mod, gtable, oracle_spline, kind, active):
    cell, periodic, r_cut = CELLS[kind]
    n = _density((9, 8, 7), cell, active)
    s = np.sort(n, axis=None)[::-1]
    _check_fp64(V, oracle_mod, gtable, oracle_spline, n, cell, periodic, 0.5 * (s[active - 1] + s[active]), r_cut)


@pytest.mark.parametrize("shape", [(4, 4), (9, 5), (70000, 60)])
def test_table_shapes_fp64(V, oracle_mod, shape):
    """The smallest table, a small one, and one too large to be kept as polynomials."""
    nD, nd = shape
    D = np.linspace(0.0, 12.0, nD)[:, None]
    dl = (np.arange(nd) / nd)[None, :]
    nodes = (1.0 - 0.3 * dl ** 2) * np.exp(-0.2 * D) * np.cos(0.3 * D) - 1e-3
    cell, periodic, r_cut = CELLS["slab"]
    n = _density((9, 8, 7), cell, 6)
    _check_fp64(V, oracle_mod, V.Table.from_nodes(nodes, 12.0), oracle_mod.Spline(nodes, 12.0), n, cell, periodic,
                1e-6, r_cut)


def test_displacements_beyond_a_table_fp64(V, oracle_mod, gtable, oracle_spline):
    """Three points and a cutoff so long that the index displacements fill no table."""
    cell = np.diag((5.0, 4.4, 8.0))
    n = _density((9, 8, 7), cell, 8)
    s = np.sort(n, axis=None)[::-1]
    _check_fp64(V, oracle_mod, gtable, oracle_spline, n, cell, (True, True, True), 0.5 * (s[2] + s[3]), 150.0)


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-6), ("fp64", 1e-12)])
def test_orthogonal_beside_skewed_in_a_batch(V, gtable, precision, tol):
    """Orthogonal and skewed cells in one batched launch give the single calls' energies."""
    kinds = ["slab", "skew", "slab"]
    ns = [_t(_density((9 + k, 8, 7), CELLS[c][0], k)) for k, c in enumerate(kinds)]
    geo = [CELLS[c][0] if c == "skew" else np.diag(CELLS[c][0]) for c in kinds]
    per = [CELLS[c][1] for c in kinds]
    E, _ = V.energy_batched(ns, geo, per, 1e-6, 6.0, gtable, precision)
    for n, g, p, e in zip(ns, geo, per, E):
        one, _ = V.energy(n, g, p, 1e-6, 6.0, gtable, precision)
        assert abs(e - one) <= tol * abs(one)


@pytest.mark.parametrize("active", [1, 33, 64, 65, 129])
def test_skewed_open_cell(V, oracle_mod, gtable, oracle_spline, active):
    """A skewed cell without images or a cutoff (its own instance of the FP32 kernel), and
    the same with a cutoff beyond every distance (the general one)."""
    cell = CELLS["skew"][0]
    n = _density((9, 8, 7), cell, active)
    s = np.sort(n, axis=None)[::-1]
    n_cut = 0.5 * (s[active - 1] + s[active])
    for r_cut in (0.0, 60.0):
        _check(V, oracle_mod, gtable, oracle_spline, n, cell, (False, False, False), n_cut, r_cut)


@pytest.mark.parametrize("active", [1, 33, 64, 65, 129])
def test_open_cell_tuned_threads(V, oracle_mod, gtable, oracle_spline, active):
    """An open orthogonal cell at the thread count that has an instance for such cells
    besides the default's."""
    cell, periodic, r_cut = CELLS["open"]
    n = _density((9, 8, 7), cell, active)
    s = np.sort(n, axis=None)[::-1]
    _check(V, oracle_mod, gtable, oracle_spline, n, cell, periodic, 0.5 * (s[active - 1] + s[active]), r_cut,
           tuning={"threads": 512, "smem_row0": -1})
