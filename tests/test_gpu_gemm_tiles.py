"""BF16 products at the edges of the tile widths and of the ring stages.

The tile is 64, 128 or 256 columns wide by the number of tile pairs, a ring
stage holds one or two 64-deep tiles of the contraction, and the three
operand orders (NT forward, NN back through a weight, TN weight gradient) take
their own loads.  NT is checked exactly on small integers (every partial sum
is below 2^24); NN and TN through the loss gradients against the FP64 oracle
with BF16-rounded weights, to 3e-2 of each block's norm: each BF16 rounding on
the path is at most 2^-9, and independent ones add in quadrature.
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


@pytest.mark.parametrize("M,N,K", [
    (1, 63, 8), (129, 64, 56), (127, 65, 64), (257, 127, 72), (385, 129, 128), (256, 257, 136), (64, 1, 904),
    (17 * 256 + 1, 385, 200), (17 * 256 - 130, 512, 264),      # 128 columns, past one pair
    (33 * 256 - 127, 513, 72), (8192, 1000, 328), (77 * 256, 250, 8),  # 256 columns, several tiles a CTA
])
def test_product_is_exact_at_tile_edges(env, M, N, K):
    torch, S = env
    rng = np.random.default_rng(M + N + K)
    A, B = rng.integers(-8, 9, (M, K)), rng.integers(-8, 9, (N, K))
    to = lambda a: torch.from_numpy(a.astype(np.float32)).to(torch.bfloat16).cuda().contiguous()
    C = S.gemm_bf16(to(A), to(B)).cpu().numpy()
    assert np.array_equal(C.astype(np.float64), A.astype(np.float64) @ B.T.astype(np.float64))


@pytest.mark.parametrize("n,hidden,M", [(9, 128, 8), (12, 384, 132), (75, 512, 36), (75, 1024, 12)])
def test_weight_gradients_at_tile_widths(env, n, hidden, M):
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
        model.loss_grads(torch.from_numpy(x).cuda(), torch.from_numpy(E).cuda(), torch.from_numpy(F).cuda(), lam=0.8)
        got = model.get_grads()
        _, want = omlp.loss_and_grads(q, x.astype(np.float64), E, F.astype(np.float64), 0.8)
        for k in ("W1", "b1", "W2", "b2", "w3"):
            assert np.linalg.norm(got[k] - want[k]) <= 3e-2 * np.linalg.norm(want[k]), k
    finally:
        model.close()
