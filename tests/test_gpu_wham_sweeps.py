"""The two sweep paths of pamd_wham against the FP64 oracle.

Sizes at the edges of the table path's blocks (16 bins by 16 temperature
groups, 256 bin threads), empty bins and empty rows, and energies so large
that beta |E| passes 1e7, where the exponentials are evaluated instead.  Both
paths sum FP64 terms relative to the largest, so ln Z and ln g agree with the
oracle to rounding: a few ulp of |beta E| + |ln Z| per sweep.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
KB = 0.008314462618


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import wham as ow
    from paper_1806_06016_gb300 import build, pamd
    build.build()
    pamd.load()
    return torch, pamd, ow


def _both(env, E, T, n_bins, **kw):
    torch, pamd, ow = env
    dev = torch.from_numpy(np.ascontiguousarray(E)).cuda()
    rng = kw.pop("e_range", None)
    g = pamd.pamd_wham(dev.data_ptr(), E.shape[0], E.shape[1], T, n_bins, e_range=rng, want_hist=True, **kw)
    lo, hi = rng if rng else (None, None)
    return g, ow.wham(E, T, n_bins, e_min=lo, e_max=hi, **kw)


def _same(g, o, atol):
    np.testing.assert_array_equal(g["hist"], o["hist"])
    assert g["iterations"] == o["iterations"]
    np.testing.assert_allclose(g["lnZ"], o["lnZ"], rtol=0, atol=atol)
    fin = np.isfinite(o["ln_g"])
    np.testing.assert_array_equal(np.isfinite(g["ln_g"]), fin)
    np.testing.assert_allclose(g["ln_g"][fin], o["ln_g"][fin], rtol=0, atol=atol)
    np.testing.assert_allclose(g["lnZ_eval"], o["lnZ_eval"], rtol=0, atol=atol)
    np.testing.assert_allclose(g["e_mean_eval"], o["e_mean_eval"], rtol=1e-11)
    np.testing.assert_allclose(g["e_var_eval"], o["e_var_eval"], rtol=1e-9)


@pytest.mark.parametrize("n_temps,n_bins", [(1, 1), (2, 15), (15, 16), (16, 17), (17, 255), (33, 257), (101, 4096),
                                            (40, 4097)])
def test_table_path_edges(env, n_temps, n_bins):
    T = np.geomspace(900.0, 300.0, n_temps)
    rng = np.random.default_rng(n_temps + n_bins)
    E = np.stack([rng.gamma(40.0, KB * t, 700) for t in T]) - 2200.0
    g, o = _both(env, E, T, n_bins, max_iter=25, tol=0.0, T_eval=[850.0, 400.0])
    # |beta E| up to 900: 25 sweeps of a few 1e-13
    _same(g, o, 1e-10)


def test_empty_row_and_start_values(env):
    T = np.array([600.0, 500.0, 400.0])
    rng = np.random.default_rng(4)
    E = np.stack([rng.gamma(40.0, KB * t, 900) for t in T])
    E[1] = 1e6  # every sample of this temperature outside the range
    g, o = _both(env, E, T, 120, e_range=(50.0, 400.0), lnZ_init=[2.0, -700.0, -1500.0], max_iter=12, tol=0.0,
                 T_eval=[550.0])
    assert g["hist"][1].sum() == 0
    _same(g, o, 1e-9)


@pytest.mark.parametrize("scale", [1.0, 1e7, 1e9])
def test_large_energies(env, scale):
    """beta |E| = 2.4e2, 2.4e9 and 2.4e11 at the lowest temperature: the table and the evaluated path."""
    T = np.array([500.0, 400.0, 300.0])
    rng = np.random.default_rng(8)
    E = -600.0 * scale + np.stack([rng.gamma(20.0, KB * t, 400) for t in T]) * scale
    g, o = _both(env, E, T, 33, max_iter=3, tol=0.0, T_eval=[450.0])
    _same(g, o, 1e-11 * scale)
