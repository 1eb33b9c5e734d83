"""Resampling at the edges of its one-launch form (chunks of 512, 1024 and 2048
replicas in up to eight CTAs, 16384 replicas at most), just above it, and over
several blocks of the separate launches.

Counts, families and energies are integer work or copies: exact.  ln Q is an
FP64 sum in another order than the oracle's: 1e-12 relative.
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


@pytest.mark.parametrize("rule", [0, 1])
@pytest.mark.parametrize("R,spread", [(1, 10.0), (31, 30.0), (511, 30.0), (512, 1e5), (513, 30.0), (2049, 0.0),
                                      (4096, 30.0), (4097, 2000.0), (8192, 30.0), (8193, 30.0), (16383, 60.0),
                                      (16384, 1e4), (16385, 30.0), (49153, 1e4), (262144, 0.0), (262145, 60.0)])
def test_two_resamplings(lib, orc, R, spread, rule):
    from oracle import adaptive as oa
    n, seed = 3, 17 + R
    top = pi.make_chain(n, 2)
    x = pi.perturbed_positions(top, R, 0.02, 5)
    v = pi.gaussian_velocities(R, n, 0.5, 6)
    E = pi.random_energies(R, -50.0, spread, 8)
    fam = (np.arange(R, dtype=np.int32) * 5 + 1) % R
    ctx = lib.pamd_init(top, R, 700.0, seed, lib.torch_options(resample_rule=rule))
    try:
        lib.pamd_set_state(ctx, x, v, E, fam)
        total = 0.0
        for i, (Tp, Tn) in enumerate([(700.0, 640.0), (640.0, 600.0)], start=1):
            cnt, lnq = lib.pamd_resample(ctx, Tp, Tn)
            lnq_o, W = orc.resample_weights(E, Tp, Tn)
            want = (oa.systematic_counts if rule else orc.multinomial_counts)(W, seed, i)
            np.testing.assert_array_equal(cnt, want)
            assert abs(lnq - lnq_o) <= 1e-12 * max(1.0, abs(lnq_o))
            E, fam, total = np.repeat(E, want), np.repeat(fam, want), total + lnq_o
            _, _, eg, fg = lib.pamd_get_state(ctx, positions=False, velocities=False)
            np.testing.assert_array_equal(eg, E)
            np.testing.assert_array_equal(fg, fam)
            o = lib.pamd_observables(ctx, Tn)
            assert o["max_copies"] == want.max() and o["R_live"] == R
        assert abs(o["sum_lnQ"] - total) <= 1e-12 * max(1.0, abs(total))
    finally:
        lib.pamd_destroy(ctx)


@pytest.mark.parametrize("R", [700, 9000])
def test_non_finite_energies_get_no_copies(lib, orc, R):
    top = pi.make_chain(3, 2)
    E = pi.random_energies(R, -50.0, 20.0, 8)
    E[[0, R // 2]] = np.inf, np.nan
    x = pi.perturbed_positions(top, R, 0.02, 5)
    ctx = lib.pamd_init(top, R, 700.0, 3, lib.torch_options())
    try:
        lib.pamd_set_state(ctx, x, np.zeros_like(x), E, np.arange(R, dtype=np.int32))
        with pytest.raises(lib.PamdError) as err:
            lib.pamd_resample(ctx, 700.0, 640.0)
        assert err.value.code == lib.PAMD_ENONFINITE
        fam = lib.pamd_get_state(ctx, positions=False, velocities=False)[3]
        assert not np.isin([0, R // 2], fam).any()
    finally:
        lib.pamd_destroy(ctx)
