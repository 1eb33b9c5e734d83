"""pamd_mlp_fit_normalization against numpy in 64 bits.

Sizes around the kernels' tiles and slices (a tile is 24 KB of positions, a
block 256 pairs).  mu and sd are FP32 results of sums that carry about 44
bits: each deviation is rounded once to FP32 (2^-24, unbiased, averaged over
the samples) and the result once more, so 2 x 2^-24 = 1.2e-7 bounds the
relative error; the tests allow 2.5e-7.
"""
import numpy as np
import pytest

import pamd_inputs as pi

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("n,M", [(2, 2), (9, 3), (24, 63), (24, 64), (24, 65), (75, 20), (75, 1777), (75, 20000),
                                 (129, 300), (256, 13)])
def test_statistics_match_64_bits(env, n, M):
    x = pi.perturbed_positions(pi.make_chain(n, 3), M, 0.01, M).astype(np.float32)
    E = np.random.default_rng(M).normal(-2000.0, 30.0, M)
    p = _fit(env, x, E)
    i, j = np.triu_indices(n, 1)
    s = q = 0.0
    d = x.astype(np.float64)
    first = 1.0 / np.linalg.norm(d[0, i] - d[0, j], axis=-1)
    for c in np.array_split(d, max(1, M // 500)):
        g = 1.0 / np.linalg.norm(c[:, i] - c[:, j], axis=-1) - first
        s, q = s + g.sum(0), q + (g * g).sum(0)
    mu, sd = first + s / M, np.sqrt(q / M - (s / M) ** 2)
    assert np.max(np.abs(p["mu"] - mu) / mu) <= 2.5e-7
    assert np.max(np.abs(p["sd"] - sd) / sd) <= 2.5e-7
    assert abs(p["mu_E"] - E.mean()) <= 1e-13 * abs(E.mean())
    assert abs(p["sigma_E"] - E.std()) <= 1e-12 * E.std()


def test_constant_and_coincident_pairs(env):
    """A zero deviation becomes 1; a pair of coincident atoms takes the FP64 path (mean inf, deviation 1),
    and neither touches the other pairs."""
    x = np.repeat(pi.make_chain(6, 3).x0[None].astype(np.float32), 90, 0)
    x[:, 5] += np.linspace(0.0, 0.01, 90, dtype=np.float32)[:, None]
    x[7, 1] = x[7, 0]
    p = _fit(env, x, np.zeros(90))
    i, j = np.triu_indices(6, 1)
    with np.errstate(divide="ignore"):
        g = 1.0 / np.linalg.norm(x.astype(np.float64)[:, i] - x.astype(np.float64)[:, j], axis=-1)
    assert p["sigma_E"] == 1.0 and p["mu_E"] == 0.0
    for k in range(len(i)):
        if (i[k], j[k]) == (0, 1):
            assert np.isinf(p["mu"][k]) and p["sd"][k] == 1.0
        elif 1 not in (i[k], j[k]) and j[k] != 5:
            assert p["sd"][k] == 1.0 and abs(p["mu"][k] - g[0, k]) <= 2.5e-7 * g[0, k]
        else:
            assert abs(p["mu"][k] - g[:, k].mean()) <= 2.5e-7 * g[:, k].mean()
            assert abs(p["sd"][k] - g[:, k].std()) <= 2.5e-7 * g[:, k].std()
