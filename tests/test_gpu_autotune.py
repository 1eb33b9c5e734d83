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


def _block_seconds(pop, steps=400):
    """Best of five propagate blocks, by the host's clock: the population has a stream of its own."""
    import time
    import torch
    best = 1e9
    for _ in range(5):
        torch.cuda.synchronize()
        start = time.perf_counter()
        pop.propagate(steps, 0.001, 600.0)
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - start)
    return best


@pytest.mark.parametrize("n,R", [(22, 256), (75, 300), (12, 64)])
def test_tuned_is_not_slower_than_default(lib, n, R):
    """The default is among the shapes timed, so that the choice is at most as
    slow as the default (a tenth is left for the timing)."""
    with lib.Population(pi.make_chain(n, 1), R, 600.0, 3, lib.torch_options()) as pop:
        default = _block_seconds(pop)
        pop.autotune(100)
        assert _block_seconds(pop) <= 1.1 * default


def test_cached_shapes(lib, tmp_path, monkeypatch):
    """A file entry written before the two-warp kernel was timed does not
    stand for such a population; one written since does, and the kernel it
    names gives the default's trajectories."""
    top, path = pi.make_chain(22, 1), tmp_path / "shapes"
    monkeypatch.setenv("PAMD_TUNE_CACHE", str(path))
    path.write_text("22 255 1 0 0 8 4 2\n")
    with lib.Population(top, 255, 600.0, 3, lib.torch_options()) as pop:
        assert pop.autotune(20)["from_cache"] == 0
    line = path.read_text().splitlines()[-1].split()
    assert line[:5] == "22 255 1 0 0".split()
    # 8 lanes, 2 warps, the two-warp variant
    path.write_text("22 254 1 0 0 8 2 13\n")
    got = []
    for tune in (False, True):
        with lib.Population(top, 254, 600.0, 3, lib.torch_options()) as pop:
            if tune:
                t = pop.autotune(20)
                assert (t["from_cache"], t["lanes_per_replica"], t["warps_per_block"]) == (1, 8, 2)
                assert t["pair_arith"] == lib.PAMD_PAIRS_PACKED
            pop.propagate(30, 0.001, 600.0)
            got.append(pop.state())
    for u, w in zip(*got):
        np.testing.assert_array_equal(u, w)
