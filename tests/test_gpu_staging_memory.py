"""Device memory a context keeps after its state calls: at most 64 MiB, over
all molecules for a batch."""
import numpy as np
import pytest

import pamd_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("molecules", [1, 3])
def test_bounded_staging(molecules):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06016_gb300 import build, pamd as lib
    build.build()
    lib.load()
    R, tops = 25000, [pi.make_chain(60 + 15 * m, 1) for m in range(molecules)]  # 36 to 54 MB an array
    opt = lib.torch_options()
    inner, held = opt._allocator, {}

    def take(b, u):
        p = inner._alloc(b, u)
        held[p] = b
        return p

    def give(p, u):
        held.pop(p)
        inner._free(p, u)

    callbacks = opt.dev_alloc, opt.dev_free = lib.ALLOC_FN(take), lib.FREE_FN(give)
    if molecules == 1:
        ctx = lib.pamd_init(tops[0], R, 300.0, 1, opt)
        subs = [ctx]
    else:
        ctx = lib.pamd_init_batch(tops, [R] * molecules, [300.0] * molecules, 1, opt)
        subs = [lib.pamd_batch_sub(ctx, m) for m in range(molecules)]
    try:
        before = sum(held.values())
        for m, sub in enumerate(subs):
            x = pi.perturbed_positions(tops[m], R, 0.005, 3 + m)
            lib.pamd_set_state(sub, x, 0.5 * x)
            got = lib.pamd_get_state(sub)
            np.testing.assert_array_equal(got[0], x.astype(np.float32))
            np.testing.assert_array_equal(got[1], (0.5 * x).astype(np.float32))
        assert 0 < sum(held.values()) - before <= 64 << 20
    finally:
        lib.pamd_destroy(ctx)
    assert not held and callbacks
