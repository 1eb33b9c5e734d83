"""Pair passes of the surrogate, two configurations at a time.

A configuration's energy and forces must not depend on its partner, on the
batch size (one, two or eight configurations to a block) or on the batch's
last odd one: equal bit for bit.  Forces against the FP64 oracle with
BF16-rounded weights, over the sizes where the row sums split differently and
at the limit of the matrix form, to 2e-2 of the RMS force (BF16 roundings of
2^-9 each on a path of three layers); loss gradients to 3e-2 of each block's
norm, as two more products lie on their path.  MD steps: a replica's path does
not depend on its partner or on an odd last one, bit for bit, and follows the
oracle's to 1e-4 nm (a relative force error of 2e-2 at the 1e4 kJ/mol/nm of
this model moves 1 u by 2e-4 (dt theta)^2 = 1.8e-9 x 1e4 nm in three steps).
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


@pytest.mark.parametrize("n", [4, 21, 22, 31, 42, 43, 48, 49, 82, 83, 97, 128, 129])
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


@pytest.mark.parametrize("n", [31, 48, 97, 128, 130])
def test_loss_gradients_over_the_row_splits(env, n):
    torch, S = env
    M = 8
    x = pi.perturbed_positions(pi.make_chain(n, 4), M, 0.02, 2).astype(np.float32)
    model, q = _model(S, n, x)
    try:
        rng = np.random.default_rng(M)
        E = -40.0 + 15.0 * rng.normal(0, 1, M)
        F = rng.normal(0, 200.0, (M, n, 3)).astype(np.float32)
        loss = model.loss_grads(torch.from_numpy(x).cuda(), torch.from_numpy(E).cuda(), torch.from_numpy(F).cuda(), lam=0.8)
        got = model.get_grads()
        want_loss, want = omlp.loss_and_grads(q, x.astype(np.float64), E, F.astype(np.float64), 0.8)
        assert abs(loss - want_loss) <= 3e-2 * abs(want_loss)
        for k in ("W1", "b1", "W2", "b2", "w3"):
            assert np.linalg.norm(got[k] - want[k]) <= 3e-2 * np.linalg.norm(want[k]), k
    finally:
        model.close()


@pytest.mark.parametrize("n", [5, 21, 22, 42, 43, 85, 86, 128, 129])
def test_steps_at_block_sizes(env, n):
    torch, S = env
    from paper_1806_06016_gb300 import pamd
    theta, dt, T, seed = 3, 0.001, 600.0, 31
    top = pi.make_chain(n, 2)
    model, q = _model(S, n, pi.perturbed_positions(top, 32, 0.03, 5).astype(np.float32))
    out = {}
    try:
        for R in (6, 7):
            ctx = pamd.pamd_init(top, R, T, seed)
            try:
                x0, v0, _, _ = pamd.pamd_get_state(ctx)
                S.attach(ctx, model)
                pamd.pamd_propagate(ctx, theta, dt, T)
                out[R] = (x0, v0) + pamd.pamd_get_state(ctx)[:3] + (pamd.pamd_observables(ctx, T),)
            finally:
                pamd.pamd_destroy(ctx)
        for a, b in zip(out[6][:5], out[7][:5]):
            np.testing.assert_array_equal(a, b[:6])
        x0, v0, x1, _, E1, obs = out[7]
        slots = np.arange(7)
        xo, _, Eo = omlp.propagate(q, x0, v0, top.mass, theta, dt, T, 1.0, seed, 0, slots=slots)
        assert np.abs(x1 - xo).max() < 1e-4
        assert np.abs(E1 - Eo).max() <= 2e-2 * q["sigma_E"]
        rg = np.sqrt(((x1 - x1.mean(1, keepdims=True)) ** 2).sum(-1).mean(1))
        assert abs(obs["rg"] - rg.mean()) <= 1e-6 * rg.mean()
    finally:
        model.close()
