"""mu and sd of pamd_mlp_fit_normalization are the FP32 roundings of 64-bit
values: half an FP32 ulp, at most 2^-24 of the value, and what the sums lose.

1/r carries 2^-44 of its value, so mu loses 2^-44 and sd, for a spread of at
least 2^-16 of the mean, 2^-28; a smaller spread is computed in FP64.  The
numpy reference loses 2^-52 of g in each deviation, 2^-29 of the smallest spread here.
"""
import numpy as np
import pytest

import pamd_inputs as pi

pytestmark = pytest.mark.gpu

MU_TOL, SD_TOL = 2.0 ** -24 + 2.0 ** -40, 2.0 ** -24 + 2.0 ** -27


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06016_gb300 import build, pamd, surrogate
    build.build()
    pamd.load()
    return torch, surrogate


def _fit(env, x, E):
    torch, S = env
    model = S.MLP(x.shape[1], 32, seed=1)
    try:
        model.fit_normalization(torch.from_numpy(x).cuda(), torch.from_numpy(E).cuda())
        return model.get_params()
    finally:
        model.close()


def _features(x):
    i, j = np.triu_indices(x.shape[1], 1)
    d = x.astype(np.float64)
    with np.errstate(divide="ignore", invalid="ignore"):
        return 1.0 / np.sqrt(((d[:, i] - d[:, j]) ** 2).sum(-1))


def _check(p, g, cols=slice(None)):
    g = g[:, cols]
    mu = g.mean(0)
    d = g - mu
    sd = np.sqrt((d * d).mean(0) - d.mean(0) ** 2)
    assert np.max(np.abs(p["mu"][cols] - mu) / mu) <= MU_TOL
    assert np.max(np.abs(p["sd"][cols] - sd) / sd) <= SD_TOL


@pytest.mark.parametrize("n,M,jitter", [(75, 2, 0.008), (75, 3, 0.008), (40, 21, 0.008), (9, 171, 0.008), (30, 2000, 0.008),
                                        (30, 500, 1e-4), (30, 500, 1e-5), (12, 300, 1e-6), (256, 7, 0.01)])
def test_rounded_64_bit_values(env, n, M, jitter):
    x = pi.perturbed_positions(pi.make_chain(n, 3), M, jitter, M + n).astype(np.float32)
    _check(_fit(env, x, np.zeros(M)), _features(x))


@pytest.mark.parametrize("far", [2.0, 30.0])
def test_first_configuration_far_from_the_rest(env, far):
    """The deviations are taken from the first configuration of a slice."""
    x = pi.perturbed_positions(pi.make_chain(20, 3), 3000, 0.005, 1).astype(np.float32)
    x[0] *= np.float32(far)
    _check(_fit(env, x, np.zeros(3000)), _features(x))


def test_non_finite_positions(env):
    """They spoil the pairs of their atoms only: mean NaN (NaN, or a difference of infinities) or that of
    1/inf = 0, deviation as numpy has it or, where that is not a number, 1."""
    n, M = 8, 100
    x = pi.perturbed_positions(pi.make_chain(n, 3), M, 0.008, 2).astype(np.float32)
    x[40, 2, 1] = np.nan
    x[63, 5, 0] = np.inf
    p = _fit(env, x, np.zeros(M))
    g = _features(x)
    i, j = np.triu_indices(n, 1)
    nan, inf = (i == 2) | (j == 2), ((i == 5) | (j == 5)) & (i != 2) & (j != 2)
    _check(p, g, ~nan & ~inf)
    assert np.all(np.isnan(p["mu"][nan])) and np.all(p["sd"][nan] == 1.0)
    _check(p, g, inf)
