"""The launch shape reported for an all-FP64 population is that of its kernel:
lanes x atoms per lane of one warp per block."""
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


# 75 atoms: 15 lanes x 5 atoms fill the chip at 2048 replicas, 25 x 3 spread 64 over it
@pytest.mark.parametrize("n,R,lanes,shape", [(75, 2048, 0, (15, 5)), (75, 64, 0, (25, 3)), (75, 64, 19, (19, 4)),
                                             (5, 9, 0, None), (256, 3, 0, (32, 8))])
def test_reported_shape(lib, n, R, lanes, shape):
    opt = lib.torch_options(precision=lib.PAMD_PREC_FP64, lanes_per_replica=lanes)
    with lib.Population(pi.make_chain(n, 1), R, 600.0, 3, opt) as pop:
        info, got, tuned = pop.info(), lib.pamd_get_shape(pop.ctx), pop.autotune(5)
    L, B = got["lanes_per_replica"], got["atoms_per_lane"]
    assert shape is None or (L, B) == shape
    assert 1 <= L <= 32 and L * B >= n
    assert (info["lanes_per_replica"], info["atoms_per_lane"], info["replicas_per_block"]) == (L, B, 32 // L)
    for s in (got, tuned):
        assert (s["lanes_per_replica"], s["atoms_per_lane"]) == (L, B)
        assert (s["warps_per_block"], s["replicas_per_lane"], s["from_cache"]) == (1, 1, 0)
        assert s["pair_arith"] == lib.PAMD_PAIRS_SCALAR
