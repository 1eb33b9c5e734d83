"""pamd_wham on a device whose free memory holds its histograms but not the
table of Boltzmann factors (24 bytes a temperature and bin): the sweeps that
evaluate every exponential need no table."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_without_memory_for_the_table():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06016_gb300 import build, pamd
    build.build()
    pamd.load()
    nT, R, bins = 600, 4096, 60000  # histograms 144 MB, table 864 MB
    T = np.geomspace(400.0, 300.0, nT)
    E = torch.from_numpy(np.random.default_rng(1).gamma(107.0, 0.00831446 * T[:, None], (nT, R))).cuda()

    def run():
        return pamd.pamd_wham(E.data_ptr(), nT, R, T, bins, max_iter=5, tol=0.0, T_eval=[350.0])

    ref = run()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    spare = 400 << 20
    hold = torch.empty(torch.cuda.mem_get_info()[0] - spare, dtype=torch.uint8, device="cuda")
    try:
        got = run()
    finally:
        del hold
        torch.cuda.empty_cache()
    # the two forms add up to 60000 64-bit terms in different orders in each of five sweeps: 60000 x 5 x 2^-53 = 3e-11
    for k in ("lnZ", "lnZ_eval", "e_mean_eval", "e_var_eval"):
        np.testing.assert_allclose(got[k], ref[k], rtol=1e-9, atol=1e-9)
    np.testing.assert_array_equal(np.isinf(got["ln_g"]), np.isinf(ref["ln_g"]))
    used = ~np.isinf(ref["ln_g"])
    np.testing.assert_allclose(got["ln_g"][used], ref["ln_g"][used], rtol=1e-9, atol=1e-9)
    assert got["iterations"] == ref["iterations"] == 5
