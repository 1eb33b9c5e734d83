"""State arrays of small populations are converted on the host: a kernel and
its staging buffer take longer there.  Exact copies on both sides of the line,
and without staging memory beyond it.
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


# one array is converted on the device from 4001 replicas x atoms on, two together from 8001
@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n,R,one,two", [(5, 800, 0, 0), (5, 801, 1, 0), (5, 1600, 1, 0), (5, 1601, 1, 1), (3, 1, 0, 0)])
def test_exact_on_both_sides(lib, n, R, one, two, fp64):
    rng = np.random.default_rng(R)
    x, v = rng.normal(0, 2, (R, n, 3)), rng.normal(0, 1, (R, n, 3))
    keep = (lambda a: a) if fp64 else (lambda a: a.astype(np.float32).astype(np.float64))
    opt = lib.torch_options(precision=lib.PAMD_PREC_FP64 if fp64 else lib.PAMD_PREC_MIXED)
    with lib.Population(pi.make_chain(n, 1), R, 300.0, 1, opt) as pop:
        n0 = lib.pamd_launch_count(pop.ctx)
        pop.set_state(x, v)
        n1 = lib.pamd_launch_count(pop.ctx)
        got = pop.state()
        n2 = lib.pamd_launch_count(pop.ctx)
        only = lib.pamd_get_state(pop.ctx, velocities=False, energies=False, families=False)
        n3 = lib.pamd_launch_count(pop.ctx)
        vel = lib.pamd_get_state(pop.ctx, positions=False, energies=False, families=False)
        bad = v.copy()
        bad[0, 0, 0] = np.inf
        with pytest.raises(lib.PamdError) as err:
            pop.set_state(2 * x, bad)
        assert err.value.code == lib.PAMD_EINVAL
        after = pop.state()
    assert (n1 - n0, n2 - n1, n3 - n2) == (two, 2 * two, one)
    for a, b in ((got[0], x), (got[1], v), (only[0], x), (vel[1], v), (after[0], x), (after[1], v)):
        np.testing.assert_array_equal(a, keep(b))


@pytest.mark.parametrize("fp64", [False, True])
def test_larger_population_without_staging_memory(lib, fp64):
    n, R = 22, 500
    top = pi.make_chain(n, 1)
    x = pi.perturbed_positions(top, R, 0.01, 3)
    v = pi.gaussian_velocities(R, n, 0.5, 4)
    out = []
    for refuse in (False, True):
        opt = lib.torch_options(precision=lib.PAMD_PREC_FP64 if fp64 else lib.PAMD_PREC_MIXED)
        inner, state = opt._allocator, {"refuse": False}
        sizes = {(s + 255) // 256 * 256 for s in (256 + 24 * n * R, 256 + 48 * n * R)}
        alloc = lib.ALLOC_FN(lambda b, u: None if state["refuse"] and b in sizes else inner._alloc(b, u))
        opt.dev_alloc = alloc
        with lib.Population(top, R, 300.0, 1, opt) as pop:
            state["refuse"] = refuse
            pop.set_state(x, v)
            out.append(pop.state() + tuple(pop.forces()))
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
