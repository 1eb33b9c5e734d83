"""The energy of a model whose hidden layer fits one 64-column tile: equal in
every bit to that of the same model padded with zero units to 128, whose
sums run in a wider tile (the padding adds exact zeros to the same order)."""
import numpy as np
import pytest

import pamd_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden", [32, 64])
@pytest.mark.parametrize("M", [1, 33, 128, 300])
def test_padded_model_has_the_same_energies(hidden, M):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06016_gb300 import build, pamd, surrogate
    build.build()
    pamd.load()
    n, rng = 9, np.random.default_rng(M)
    p, wide = n * (n - 1) // 2, 128
    small = {"W1": rng.normal(0, 0.2, (hidden, p)), "b1": rng.normal(0, 0.3, hidden),
             "W2": rng.normal(0, 0.2, (hidden, hidden)), "b2": rng.normal(0, 0.3, hidden), "w3": rng.normal(0, 0.3, hidden)}
    norm = {"b3": 0.25, "mu": np.full(p, 3.0, np.float32), "sd": np.ones(p, np.float32), "mu_E": -40.0, "sigma_E": 15.0}
    x = torch.from_numpy(pi.perturbed_positions(pi.make_chain(n, 4), M, 0.02, 2).astype(np.float32)).cuda()
    got = []
    for h in (hidden, wide):
        w = {k: np.pad(a, [(0, h - hidden if s == hidden else 0) for s in a.shape]).astype(np.float32)
             for k, a in small.items()}
        model = surrogate.MLP(n, h, seed=1)
        try:
            model.set_params({**w, **norm})
            got.append([t.cpu().numpy() for t in model.energy_forces(x)])
        finally:
            model.close()
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])
