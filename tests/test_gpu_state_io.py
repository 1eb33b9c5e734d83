"""State and force arrays through the device layout kernels: exact copies
(FP32 rounding in the mixed mode) for small, padded and chunked populations,
the host path without staging memory, and a refused state that leaves the
population as it was.
"""
import numpy as np
import pytest

import pamd_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06016_gb300 import build, pamd
    build.build()
    pamd.load()
    return pamd


def _state(n, R, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(0, 2, (R, n, 3)), rng.normal(0, 1, (R, n, 3)), rng.normal(0, 9, R), \
        rng.integers(0, R, R).astype(np.int32)


# 256 atoms x 12000 replicas: 147 MB of rows, three chunks of the 64 MB staging memory
@pytest.mark.parametrize("n,R", [(1, 1), (3, 5), (75, 1001), (256, 12000)])
@pytest.mark.parametrize("fp64", [False, True])
def test_round_trip_and_refusal(lib, n, R, fp64):
    x, v, E, fam = _state(n, R, n)
    keep = (lambda a: a) if fp64 else (lambda a: a.astype(np.float32).astype(np.float64))
    opt = lib.torch_options(precision=lib.PAMD_PREC_FP64 if fp64 else lib.PAMD_PREC_MIXED)
    with lib.Population(pi.make_chain(n, 1), R, 300.0, 1, opt) as pop:
        pop.set_state(x, v, E, fam)
        bad = x.copy()
        bad[-1, -1, -1] = np.nan
        with pytest.raises(lib.PamdError) as err:
            pop.set_state(bad, 2 * v, 2 * E, fam[::-1].copy())
        assert err.value.code == lib.PAMD_EINVAL
        xs, vs, Es, fs = pop.state()
    np.testing.assert_array_equal(xs, keep(x))
    np.testing.assert_array_equal(vs, keep(v))
    np.testing.assert_array_equal(Es, E)
    np.testing.assert_array_equal(fs, fam)


@pytest.mark.parametrize("fp64", [False, True])
def test_without_staging_memory(lib, fp64):
    n, R = 22, 333
    top = pi.make_chain(n, 1)
    x = pi.perturbed_positions(top, R, 0.01, 3)
    v = pi.gaussian_velocities(R, n, 0.5, 4)
    out = []
    for refuse in (False, True):
        opt = lib.torch_options(precision=lib.PAMD_PREC_FP64 if fp64 else lib.PAMD_PREC_MIXED)
        inner, state = opt._allocator, {"refuse": False}
        # staging memory is asked for by its size: rows of x and v or of one array, and a flag
        sizes = {(s + 255) // 256 * 256 for s in (256 + 24 * n * R, 256 + 48 * n * R)}
        alloc = lib.ALLOC_FN(lambda b, u: None if state["refuse"] and b in sizes else inner._alloc(b, u))
        opt.dev_alloc = alloc
        with lib.Population(top, R, 300.0, 1, opt) as pop:
            state["refuse"] = refuse
            pop.set_state(x, v)
            f, e = pop.forces()
            out.append(pop.state() + (f, e))
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
