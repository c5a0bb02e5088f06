"""The semilocal energies of densities that fall far below any cutoff, with gradients
that do not fall with them: points of a vanishing density add nothing, whatever the
gradient there.  Against the oracle at 1e-12 relative."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KEYS = ("Ex_lda", "Ec_lda", "Ex_pbe", "Ec_pbe", "Ex_revpbe")


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


def _gaussian(dims, L, a):
    x = np.meshgrid(*[(np.arange(d) + 0.3) / d * l - 0.5 * l for d, l in zip(dims, L)], indexing="ij")
    return 2.0 * np.exp(-a * sum(c * c for c in x))


def _check(V, oracle_mod, n, L, g, **kw):
    """The points below 1e-20 weigh nothing (n^(4/3) each): the reference leaves them out,
    as the oracle's own log(1 + 1/x) vanishes from about 1e-24 on and its H is NaN there."""
    ref = oracle_mod.semilocal(np.where(n > 1e-20, n, 0.0), L, g)
    got = V.semilocal(_t(n), L, (0, 0, 0), **kw)
    assert got["n_points"] == int((n > 0.0).sum())
    for k in KEYS:
        assert np.isfinite(ref[k]) and abs(got[k] - ref[k]) <= 1e-12 * abs(ref[k]), (k, got[k], ref[k])


@pytest.mark.parametrize("a", [0.5, 1.5, 3.0, 6.0])
def test_gaussian_with_the_fft_gradient(V, oracle_mod, a):
    """A Gaussian in a vacuum cell, down to 1e-15 .. 1e-200: the band-limited gradient
    keeps its rounding noise of 1e-17 out there."""
    dims, L = (24, 22, 26), (14.0, 13.0, 15.0)
    n = _gaussian(dims, L, a)
    g = V.gradient(_t(n), L, "spectral").cpu().numpy()
    _check(V, oracle_mod, n, L, g, gradient="spectral")


@pytest.mark.parametrize("low", [1e-39, 1e-45, 1e-60, 1e-84, 1e-86, 1e-90, 1e-120, 1e-160, 1e-250])
@pytest.mark.parametrize("slope", [0.0, 1e-60, 1e-18, 1.0, 1e30])
def test_low_densities_with_a_given_gradient(V, oracle_mod, low, slope):
    dims, L = (9, 8, 10), (6.0, 5.6, 7.0)
    rng = np.random.default_rng(7)
    n = 0.05 * np.exp(0.3 * rng.uniform(-1, 1, dims))
    g = 0.02 * rng.normal(size=(3,) + dims)
    n[2:5, 3:6, 4:8] = low
    g[:, 2:5, 3:6, 4:8] = slope
    _check(V, oracle_mod, n, L, g, grad=_t(g))


@pytest.mark.parametrize("a", [0.7, 2.0, 4.0])
def test_gaussian_with_finite_differences(V, oracle_mod, a):
    dims, L = (24, 22, 26), (14.0, 13.0, 15.0)
    n = _gaussian(dims, L, a)
    _check(V, oracle_mod, n, L, oracle_mod.gradient(n, [l / d for l, d in zip(L, dims)]))
