"""Pair passes of the surrogate, two configurations at a time.

A configuration's energy and forces must not depend on its partner, on the
batch size (one, two or eight configurations to a block) or on the batch's
last odd one: equal bit for bit.  Forces against the FP64 oracle with
BF16-rounded weights, over the sizes where the row sums split differently and
at the limit of the matrix form, to 2e-2 of the RMS force (BF16 roundings of
2^-9 each on a path of three layers).
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


def _model(S, n, x):
    model = S.MLP(n, 64, seed=n)
    p = model.get_params()
    g = omlp.features(x.astype(np.float64))
    p["mu"], p["sd"] = g.mean(0).astype(np.float32), (g.std(0) + 0.05).astype(np.float32)
    p["b3"], p["mu_E"], p["sigma_E"] = 0.25, -40.0, 15.0
    model.set_params(p)
    q = {k: (np.asarray(v, np.float64) if isinstance(v, np.ndarray) else float(v)) for k, v in model.get_params().items()}
    q["W1"], q["W2"] = _bf16(q["W1"]), _bf16(q["W2"])
    return model, q


@pytest.mark.parametrize("n", [4, 31, 48, 49, 97, 128, 129])
def test_forces_over_the_row_splits(env, n):
    torch, S = env
    x = pi.perturbed_positions(pi.make_chain(n, 4), 7, 0.02, 2).astype(np.float32)
    model, q = _model(S, n, x)
    try:
        xd = torch.from_numpy(x).cuda()
        E, F = model.energy_forces(xd)
        _, want = omlp.energy_forces(q, x.astype(np.float64))
        assert np.sqrt(np.mean((F.cpu().numpy() - want) ** 2)) <= 2e-2 * np.sqrt(np.mean(want ** 2))
        for m in (0, 3, 6):  # alone, and next to another partner
            for sl in (slice(m, m + 1), slice(max(m - 1, 0), m + 1)):
                e, f = model.energy_forces(xd[sl].contiguous())
                assert torch.equal(e[-1], E[m]) and torch.equal(f[-1], F[m])
    finally:
        model.close()


@pytest.mark.parametrize("n", [9, 130])
def test_large_batches_equal_small_ones(env, n):
    torch, S = env
    M = 4871  # odd, past the size where a block takes eight configurations
    x = np.tile(pi.perturbed_positions(pi.make_chain(n, 4), 37, 0.02, 2).astype(np.float32), (132, 1, 1))[:M]
    model, _ = _model(S, n, x[:37])
    try:
        xd = torch.from_numpy(x).cuda()
        E, F = model.energy_forces(xd)
        e, f = model.energy_forces(xd[:37].contiguous())
        assert torch.equal(E[:37], e) and torch.equal(F[:37], f)
        last = M - 1
        assert torch.equal(E[last], e[last % 37]) and torch.equal(F[last], f[last % 37])
        E2, _ = model.energy_forces(xd, forces=False)
        assert torch.equal(E, E2)
    finally:
        model.close()
