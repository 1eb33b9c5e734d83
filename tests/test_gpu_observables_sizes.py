"""Observables at the edges of their kernels, against the oracle.

Chunks of 1024 replicas, one launch up to 64 chunks and three above, families
in any order (also unsorted and repeated), one family holding everything, and
repeated observations of the same population (family stamps are not cleared
in between).  Sums are FP64 in another order than the oracle's: 1e-9 relative
for the averages, 1e-7 for the jackknife errors (differences of nearly equal
leave-one-out means), counts exact.
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


def _families(kind, R, rng):
    if kind == "one":
        return np.full(R, R // 2, np.int32)
    if kind == "sorted":
        return np.sort(rng.integers(0, R, R)).astype(np.int32)
    return rng.integers(0, R, R).astype(np.int32)


@pytest.mark.parametrize("R,kind", [(1, "any"), (2, "any"), (63, "any"), (1023, "sorted"), (1024, "one"), (1025, "any"),
                                    (65536, "any"), (65537, "sorted"), (70001, "one")])
def test_observables(lib, orc, R, kind):
    n = 4
    top = pi.make_chain(n, 2)
    rng = np.random.default_rng(R)
    x = pi.perturbed_positions(top, R, 0.02, 1).astype(np.float32).astype(np.float64)
    v = pi.gaussian_velocities(R, n, 0.7, 2).astype(np.float32).astype(np.float64)
    ctx = lib.pamd_init(top, R, 500.0, 3, lib.torch_options())
    try:
        for turn in range(3):
            fam = _families(kind, R, rng)
            lib.pamd_set_state(ctx, x, v, None, fam)
            lib.pamd_propagate(ctx, 0, 0.001, 500.0)
            o = lib.pamd_observables(ctx, 500.0)
            E = lib.pamd_get_state(ctx, positions=False, velocities=False)[2]
            want = orc.observables(top, x, v, fam, E)
            assert o["n_families"] == len(np.unique(fam)) and o["R_live"] == R
            for k in ("e_pot", "e_kin", "rg", "rg2"):
                assert abs(o[k] - want[k]) <= 1e-9 * abs(want[k]), (turn, k)
                assert abs(o[k + "_se"] - want[k + "_se"]) <= 1e-7 * abs(want[k + "_se"]) + 1e-12, (turn, k)
    finally:
        lib.pamd_destroy(ctx)
