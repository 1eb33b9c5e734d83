"""Loss gradients of the surrogate at the edges of the training kernels' tiles.

The reverse-pass kernels work on tiles of 32 samples by 64 hidden units, and
the sums over the samples run over the tiles: sizes below, at and past one
tile in each direction, against the FP64 oracle with BF16-rounded weights.
Tolerance 3e-2 relative to the norm of each block: every BF16 rounding on the
gradient path has relative error at most 2^-9, and the independently rounded
terms of each contraction add in quadrature (tests/test_gpu_mlp.py).
"""
import numpy as np
import pytest

import pamd_inputs as pi
from oracle import mlp as omlp

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


def _bf16(a):
    b = np.ascontiguousarray(a, dtype=np.float32).view(np.uint32).astype(np.uint64)
    return ((b + 0x7FFF + ((b >> 16) & 1)) & 0xFFFF0000).astype(np.uint32).view(np.float32).astype(np.float64)


@pytest.mark.parametrize("n,hidden,M", [(5, 32, 4), (9, 32, 32), (9, 64, 36), (9, 96, 68), (12, 160, 260)])
def test_gradients_at_tile_edges(env, n, hidden, M):
    torch, S = env
    x = pi.perturbed_positions(pi.make_chain(n, 4), M, 0.02, 2).astype(np.float32)
    model = S.MLP(n, hidden, seed=n + hidden)
    try:
        rng = np.random.default_rng(M)
        p = model.get_params()
        g = omlp.features(x.astype(np.float64))
        p["mu"], p["sd"] = g.mean(0).astype(np.float32), (g.std(0) + 0.05).astype(np.float32)
        p["b1"], p["b2"] = (rng.normal(0, 0.3, hidden).astype(np.float32) for _ in range(2))
        p["b3"], p["mu_E"], p["sigma_E"] = 0.25, -40.0, 15.0
        model.set_params(p)
        q = {k: (np.asarray(v, np.float64) if isinstance(v, np.ndarray) else float(v))
             for k, v in model.get_params().items()}
        q["W1"], q["W2"] = _bf16(q["W1"]), _bf16(q["W2"])
        E = -40.0 + 15.0 * rng.normal(0, 1, M)
        F = rng.normal(0, 200.0, (M, n, 3)).astype(np.float32)
        loss = model.loss_grads(torch.from_numpy(x).cuda(), torch.from_numpy(E).cuda(),
                                torch.from_numpy(F).cuda(), lam=0.8)
        got = model.get_grads()
        want_loss, want = omlp.loss_and_grads(q, x.astype(np.float64), E, F.astype(np.float64), 0.8)
        assert abs(loss - want_loss) <= 3e-2 * abs(want_loss)
        for k in ("W1", "b1", "W2", "b2", "w3"):
            assert np.linalg.norm(got[k] - want[k]) <= 3e-2 * np.linalg.norm(want[k]), k
        assert abs(got["b3"] - want["b3"]) <= 3e-2 * abs(want["b3"]) + 1e-6
    finally:
        model.close()
