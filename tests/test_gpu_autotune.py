"""What the launch-shape tuner may and may not choose."""
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


def test_tuning_one_molecule_leaves_the_batch_alone(lib):
    """The batch's launches are laid out for its molecules' shapes, so a
    molecule keeps its own and the batch its trajectories."""
    tops, R = [pi.make_chain(12, 3), pi.make_chain(60, 4)], [70, 40]
    got = []
    for tune in (False, True):
        ctx = lib.pamd_init_batch(tops, R, [900.0] * 2, 1, lib.torch_options())
        try:
            for m in range(2):
                sub = lib.pamd_batch_sub(ctx, m)
                shape = lib.pamd_get_shape(sub)
                if tune:
                    assert lib.pamd_autotune(sub, 20) == shape
                    assert lib.pamd_get_shape(sub) == shape
            lib.pamd_propagate(ctx, 20, 0.001, 900.0)
            got.append([lib.pamd_get_state(lib.pamd_batch_sub(ctx, m)) for m in range(2)])
        finally:
            lib.pamd_destroy(ctx)
    for a, b in zip(*got):
        for u, w in zip(a, b):
            np.testing.assert_array_equal(u, w)
