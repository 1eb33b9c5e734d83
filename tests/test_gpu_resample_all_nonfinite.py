"""A population without a single finite energy: every weight is 0, every draw
falls past the last cumulative weight and is taken by the last replica, in the
one-launch resampling (up to 16384 replicas) as in the separate launches."""
import numpy as np
import pytest

import pamd_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rule", [0, 1])
@pytest.mark.parametrize("R", [1, 300, 512, 4097, 16384, 20000])
def test_last_replica_takes_every_draw(R, rule):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06016_gb300 import build, pamd as lib
    build.build()
    lib.load()
    top = pi.make_chain(3, 2)
    x = pi.perturbed_positions(top, R, 0.02, 5)
    E = np.full(R, np.nan)
    E[::2] = np.inf
    with lib.Population(top, R, 700.0, 3, lib.torch_options(resample_rule=rule)) as pop:
        pop.set_state(x, np.zeros_like(x), E, np.arange(R, dtype=np.int32))
        with pytest.raises(lib.PamdError) as err:
            pop.resample(700.0, 640.0)
        assert err.value.code == lib.PAMD_ENONFINITE
        _, _, got, fam = lib.pamd_get_state(pop.ctx, positions=False, velocities=False)
        assert np.all(fam == R - 1)
        np.testing.assert_array_equal(got, np.full(R, E[R - 1]))
        # finite energies make it an ordinary population again
        pop.set_state(x, np.zeros_like(x), np.linspace(-1.0, 0.0, R), np.arange(R, dtype=np.int32))
        copies, _ = pop.resample(700.0, 640.0)
        assert copies.sum() == R
