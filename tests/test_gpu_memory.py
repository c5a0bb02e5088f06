"""What the library keeps on the device, and calls that go without an optional part of
it: the FP64 polynomials and the texture copy of a table, the scratch pool of calls
without a table, the distance tables of a large batch."""
import subprocess
import sys

import numpy as np
import pytest

from conftest import ROOT

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


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info(0)[0]


DIMS, L = (9, 8, 10), (5.0, 4.4, 5.6)


def _density(seed=1):
    return 0.05 * np.exp(0.3 * np.random.default_rng(seed).uniform(-1, 1, DIMS))


def _nodes(nD, nd):
    D = np.linspace(0.0, 12.0, nD)[:, None]
    dl = (np.arange(nd) / nd)[None, :]
    return (1.0 - 0.3 * dl ** 2) * np.exp(-0.2 * D) * np.cos(0.3 * D) - 1e-3


def test_large_table_in_fp32_has_no_polynomials(V, oracle_mod):
    """A table of 60000 x 60 nodes: 30 MB of FP64 and 15 MB of FP32 coefficients; its
    polynomials (119 MB) come with the first FP64 sum."""
    nodes = _nodes(60000, 60)
    n = _density()
    P = oracle_mod.Problem(n, L, (False,) * 3, 1e-6, 0.0, oracle_mod.Spline(nodes, 12.0))
    e = P.energy()["E"]
    t = _t(n)
    table = V.Table.from_nodes(nodes, 12.0)
    small = V.Table.from_nodes(_nodes(30, 6), 12.0)
    for prec in ("fp32", "fp64"):
        V.energy(t, L, (0, 0, 0), 1e-6, 0.0, small, prec)  # everything else is in place
    free0 = _free()
    E, _ = V.energy(t, L, (0, 0, 0), 1e-6, 0.0, table, "fp32")
    free1 = _free()
    assert abs(E - e) <= 1e-6 * abs(e)
    assert free0 - free1 < 80 << 20
    E, _ = V.energy(t, L, (0, 0, 0), 1e-6, 0.0, table, "fp64")
    assert abs(E - e) <= 1e-10 * abs(e)
    assert 100 << 20 < free1 - _free() < 160 << 20
    table.free()
    small.free()


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-6), ("fp64", 1e-10)])
def test_calls_without_the_optional_table_copies(V, oracle_mod, oracle_table, oracle_spline, monkeypatch, precision, tol):
    """When the polynomials and the texture cannot be had, the sums take the coefficients."""
    n = _density(2)
    P = oracle_mod.Problem(n, L, (True, True, False), 1e-6, 6.0, oracle_spline)
    e = P.energy()
    v = P.potential(e["A"], e["U"])
    monkeypatch.setenv("VDWDF_FAIL_ALLOC", "2")
    table = V.Table.from_nodes(oracle_table, 30.0)
    args = (_t(n), L, P.periodic, 1e-6, 6.0, table, precision)
    E, r = V.energy(*args)
    Ev, vg, rv = V.potential(*args)
    Eb, _ = V.energy_batched([args[0]], [L], [P.periodic], 1e-6, 6.0, table, precision)
    En, rn = V.energy_noalloc(*args)
    for x, res in ((E, r), (Ev, rv), (En, rn)):
        assert abs(x - e["E"]) <= tol * abs(e["E"]) and res["pairs"] == e["pairs"]
    assert abs(Eb[0] - e["E"]) <= tol * abs(e["E"])
    assert np.max(np.abs(vg.cpu().numpy() - v)) <= 10 * tol * np.max(np.abs(v))
    monkeypatch.delenv("VDWDF_FAIL_ALLOC")
    table.free()


CHILD = """
import torch
import numpy as np
import paper_0810_2273_gb300 as V
def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info(0)[0]
n = torch.full((120, 120, 120), 0.05, dtype=torch.float64, device="cuda:0")
table = V.Table.from_nodes(np.linspace(1.0, 0.1, 24).reshape(6, 4), 12.0)
calls = (lambda: V.semilocal(n, (60.0,) * 3, (1, 1, 1), gradient="spectral"),
         lambda: V.far_tail(n, (60.0,) * 3, (1, 1, 1), 1e-6, 8.0, want_v=True),
         lambda: V.far_tail(n, (60.0,) * 3, (1, 0, 0), 1e-6, 8.0))
for call in calls:
    call()
with_table = free()
table.free()
without = free()
print(without - with_table)
for call in calls:
    for _ in range(2):
        call()
        print(without - free())
"""


def test_scratch_is_given_back_without_tables():
    """Semilocal energies and far fields, which take no table, keep no device memory
    when they return while no table lives (in a process of its own)."""
    out = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, cwd=ROOT, timeout=600)
    assert out.returncode == 0, out.stderr[-2000:]
    kept = [int(x) for x in out.stdout.split()]
    assert kept[0] >= 32 << 20  # what the calls kept while the table lived
    assert kept[1:] == [0] * 6, kept


def test_large_fp64_batch_bounds_its_distance_tables(V, oracle_mod, oracle_table, oracle_spline):
    """Two hundred cells of two active points under a long cutoff, whose tables of
    distances (55 MB each) would take 11 GB: the batch takes them for as many as fit
    its bound and computes the others' distances; all energies agree."""
    table = V.Table.from_nodes(oracle_table, 30.0)
    base = np.zeros(DIMS)
    base[2, 3, 4], base[5, 6, 1] = 0.3, 0.2
    ns = [_t(base * (1.0 + 0.001 * k)) for k in range(200)]
    per, rc = (True, True, True), 105.0
    V.energy_batched(ns[:1], [L], [per], 1e-6, 20.0, table, "fp64")
    free0 = _free()
    E, r = V.energy_batched(ns, [L] * 200, [per] * 200, 1e-6, rc, table, "fp64")
    assert free0 - _free() < 2 << 30
    for k in (0, 18, 19, 199):
        e = oracle_mod.Problem(base * (1.0 + 0.001 * k), L, per, 1e-6, rc, oracle_spline).energy()
        assert abs(E[k] - e["E"]) <= 1e-10 * abs(e["E"])
    assert r["pairs"] == 200 * e["pairs"]
    table.free()
