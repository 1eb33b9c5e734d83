"""Two-warp propagate kernel against the one-warp kernel, bit for bit.

Small populations of linear chains run the pairs of a step and the rest of it
in two warps; an explicit block size keeps the one-warp kernel.  Both apply
the same FP32 instructions in the same order, so states, energies and
observables must be equal in every bit: for 3 to 8 atoms per lane (8 has no
two-warp form), full and partial replica groups, odd and even lane counts
(with the antipodal tile), a theta of 0, and a population past the limit.
"""
import numpy as np
import pytest

import pamd_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pamd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06016_gb300 import build, pamd as mod
    build.build()
    mod.load()
    return mod


@pytest.mark.parametrize("n,R", [(10, 1), (12, 37), (22, 5), (22, 256), (31, 33), (36, 41), (47, 3), (75, 2), (75, 61),
                                 (90, 7), (110, 9), (130, 12), (150, 31), (170, 6), (200, 17), (224, 5), (250, 3),
                                 (75, 700)])
def test_split_equals_one_warp(pamd, n, R):
    top = pi.make_chain(n, 1)
    got = []
    for warps in (0, 4):
        o = pamd.torch_options()
        o.warps_per_block = warps
        with pamd.Population(top, R, 900.0, 11, o) as p:
            p.propagate(0, 0.001, 900.0)
            e0 = p.state()[2].copy()
            p.propagate(17, 0.001, 900.0)
            p.propagate(4, 0.001, 850.0)
            ob = p.observables(850.0)
            got.append([e0, *p.state()[:3], np.array([ob["e_kin"], ob["rg"]])])
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
