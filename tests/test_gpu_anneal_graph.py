"""What a captured anneal holds by value: a context whose graph is replayed
must give what a fresh context gives, bit for bit."""
import numpy as np
import pytest

import pamd_inputs as pi

pytestmark = pytest.mark.gpu

TEMPS, THETA, DT = [900.0, 860.0, 820.0], 7, 0.001


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06016_gb300 import build, pamd
    build.build()
    pamd.load()
    return pamd


def _run(lib, ctx):
    """Averages of an anneal and the state it leaves."""
    obs = lib.pamd_anneal(ctx, TEMPS, THETA, DT)
    subs = [lib.pamd_batch_sub(ctx, m) for m in range(max(0, lib.pamd_batch_size(ctx)))] or [ctx]
    return obs, [lib.pamd_get_state(s) for s in subs]


def _equal(a, b):
    assert a[0] == b[0]
    for p, q in zip(a[1], b[1]):
        for u, w in zip(p, q):
            np.testing.assert_array_equal(u, w)


@pytest.mark.parametrize("fp64", [False, True])
def test_another_seed_after_a_reset(lib, fp64):
    top, R = pi.make_chain(12, 2), 70
    opt = lib.torch_options(precision=lib.PAMD_PREC_FP64 if fp64 else lib.PAMD_PREC_MIXED)
    ref = {}
    for seed in (5, 6):
        with lib.Population(top, R, TEMPS[0], seed, opt) as p:
            ref[seed] = _run(lib, p.ctx)
    with lib.Population(top, R, TEMPS[0], 5, opt) as p:
        _run(lib, p.ctx)
        for seed in (6, 5, 6):
            p.reset(TEMPS[0], seed)
            _equal(_run(lib, p.ctx), ref[seed])


def test_restored_seed(lib, tmp_path):
    top, R, path = pi.make_chain(12, 2), 70, str(tmp_path / "p.ckpt")
    with lib.Population(top, R, TEMPS[0], 8) as p:
        p.checkpoint(path)
        ref = _run(lib, p.ctx)
    with lib.Population(top, R, TEMPS[0], 9) as p:
        _run(lib, p.ctx)
        p.restore(path)
        got = _run(lib, p.ctx)
    # a checkpoint does not hold what the resampling before it reported
    for obs in (got[0], ref[0]):
        del obs[0]["lnQ"], obs[0]["max_copies"]
    _equal(got, ref)


def test_batch_seeds(lib):
    """All molecules reset to another seed, then one of them alone."""
    tops, R = [pi.make_chain(12, 3), pi.make_chain(20, 4)], [70, 40]

    def fresh(resets):
        ctx = lib.pamd_init_batch(tops, R, [TEMPS[0]] * 2, 1, lib.torch_options())
        try:
            for m, seed in resets:
                lib.pamd_reset(ctx if m is None else lib.pamd_batch_sub(ctx, m), TEMPS[0], seed)
            return _run(lib, ctx)
        finally:
            lib.pamd_destroy(ctx)

    ctx = lib.pamd_init_batch(tops, R, [TEMPS[0]] * 2, 1, lib.torch_options())
    try:
        _run(lib, ctx)
        lib.pamd_reset(ctx, TEMPS[0], 2)
        _equal(_run(lib, ctx), fresh([(None, 2)]))
        lib.pamd_reset(ctx, TEMPS[0], 2)
        lib.pamd_reset(lib.pamd_batch_sub(ctx, 1), TEMPS[0], 3)
        _equal(_run(lib, ctx), fresh([(None, 2), (1, 3)]))
    finally:
        lib.pamd_destroy(ctx)


def test_force_model_at_a_freed_models_address(lib):
    """A model made after another was destroyed often takes its host address;
    the anneal captured with the first must not stand for the second."""
    import torch
    from paper_1806_06016_gb300 import surrogate
    n, R = 12, 70
    top = pi.make_chain(n, 2)

    def anneal(p, model):
        p.reset(TEMPS[0], 5)
        surrogate.attach(p.ctx, model)
        got = _run(lib, p.ctx)
        surrogate.attach(p.ctx, None)
        return got

    with lib.Population(top, R, TEMPS[0], 5, lib.torch_options()) as p, \
            lib.Population(top, R, TEMPS[0], 5, lib.torch_options()) as q:
        first = surrogate.MLP(n, 64, seed=1)
        a = anneal(p, first)
        first.close()
        hold = torch.empty(32 << 20, dtype=torch.uint8, device="cuda")  # the device memory it gave back is taken
        second = surrogate.MLP(n, 64, seed=2)
        b = anneal(p, second)
        _equal(b, anneal(q, second))
        assert not np.array_equal(a[1][0][0], b[1][0][0])
        second.close()
        del hold


def test_batch_after_a_longer_anneal_of_one_molecule(lib):
    """The longer anneal moves that molecule's observables buffer."""
    ctx = lib.pamd_init_batch([pi.make_chain(12, 3), pi.make_chain(20, 4)], [70, 40], [TEMPS[0]] * 2, 1, lib.torch_options())
    try:
        first = _run(lib, ctx)
        lib.pamd_anneal(lib.pamd_batch_sub(ctx, 0), np.linspace(900.0, 700.0, 9), THETA, DT)
        lib.pamd_reset(ctx, TEMPS[0], 1)
        again = _run(lib, ctx)
        for obs in (first[0], again[0]):  # a reset does not clear what the last resampling reported
            for o in obs[0]:
                del o["lnQ"], o["max_copies"]
        _equal(again, first)
    finally:
        lib.pamd_destroy(ctx)
