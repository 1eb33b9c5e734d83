"""The all-FP64 kernel over its shapes: lanes per replica, replicas per warp,
odd and even rings (the antipodal tile), idle lanes, padding atoms, a partly
filled last warp, and bonded terms in an order that is not a chain's.

Every operation is binary64, so forces agree with the oracle to rounding
(1e-10 relative RMS: pair forces of opposite sign cancel by a few digits) and
ten steps of a trajectory stay within 1e-10 nm, as in tests/test_gpu_fp64.py.
"""
import numpy as np
import pytest

import pamd_inputs as pi

pytestmark = pytest.mark.gpu
KB = 0.008314462618


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06016_gb300 import build, pamd
    build.build()
    pamd.load()
    return pamd


def _relabel(top, seed):
    new = np.random.default_rng(seed).permutation(top.n_atoms).astype(np.int32)
    old = np.argsort(new)
    for k in ("mass", "charge", "sigma", "epsilon", "x0"):
        setattr(top, k, getattr(top, k)[old])
    for k in ("bond", "angle", "dihedral", "excl", "pair14"):
        setattr(top, k, new[getattr(top, k)])
    return top


# n atoms, lanes (0: chosen for the population), replicas, relabelled
CASES = [(2, 0, 1, False), (3, 1, 33, False), (8, 1, 40, False), (9, 0, 2048, False), (22, 11, 5, False),
         (22, 22, 3, False), (31, 16, 3, True), (40, 8, 9, False), (75, 0, 64, False), (75, 15, 5, True),
         (75, 16, 3, False), (75, 10, 4, False), (75, 32, 2, False), (100, 13, 5, True), (128, 0, 2, False),
         (256, 32, 1, False)]


@pytest.mark.parametrize("n,lanes,R,relabelled", CASES)
def test_forces_and_steps(lib, orc, n, lanes, R, relabelled):
    top = pi.make_chain(n, 400 + n)
    top.dih_phase = np.linspace(0.2, 2.1, len(top.dih_phase))
    top.dih_n = (np.arange(len(top.dih_n)) % 6 + 1).astype(np.int32)
    if relabelled:
        top = _relabel(top, n)
    x = pi.perturbed_positions(top, R, 0.004, n)
    v = pi.gaussian_velocities(R, n, 0.6, n + 1)
    o = lib.pamd_options_default()
    o.precision = lib.PAMD_PREC_FP64
    o.lanes_per_replica = lanes
    T, dt, seed = 400.0, 0.001, 77
    ctx = lib.pamd_init(top, R, T, seed, o)
    try:
        lib.pamd_set_state(ctx, x, v)
        f, e = lib.pamd_forces(ctx)
        lib.pamd_propagate(ctx, 10, dt, T)
        xg, vg, eg, _ = lib.pamd_get_state(ctx)
    finally:
        lib.pamd_destroy(ctx)
    t = orc.Topo(top)
    for k in sorted({0, R // 2, R - 1}):
        eo, fo, terms = orc.energy_forces(t, x[k])
        rms = np.sqrt(np.mean(fo ** 2))
        assert np.sqrt(np.mean((f[k] - fo) ** 2)) <= 1e-10 * max(rms, 1e-12)
        assert abs(e[k] - eo) <= 1e-10 * max(np.abs(terms).sum(), 1e-12)
        xo, vo, _ = orc.propagate(top, x[k:k + 1], v[k:k + 1], 10, dt, T, 1.0, seed, 0, slots=np.array([k]))
        assert np.max(np.abs(xg[k] - xo[0])) <= 1e-10
        assert np.max(np.abs(vg[k] - vo[0])) <= 1e-8
        xs = xo[0]
        ee, _, terms = orc.energy_forces(t, xs)
        assert abs(eg[k] - ee) <= 1e-8 * max(np.abs(terms).sum(), 1e-12)
