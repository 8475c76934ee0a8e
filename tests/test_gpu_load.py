"""SFT loads with a bin that is not finite: refused, with its index for host
data, wherever it lies, and the context keeps what it held."""
import numpy as np
import pytest

from workload import config_mid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bins", [200, 201, 203])
@pytest.mark.parametrize("at", [0, 1, 777, -1])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_bad_bin_is_refused_and_the_context_kept(lib, n_bins, at, bad):
    import torch
    w = config_mid(seed=3, n_sft=9, n_sky=1, n_f=10, n_fdot=1, n_bins=n_bins)
    d = w.detectors[0]
    g = lib.FStat(0, dterms=w.dterms, topk=5)
    try:
        g.load_workload(w)
        g.compute()
        before = g.twoF()
        x = np.ascontiguousarray(np.stack([d.bins.real, d.bins.imag], -1), np.float32)
        flat = x.reshape(-1)
        i = at % flat.size
        flat[i] = bad
        args = (g.ctx, 0, d.lat, d.lon, d.az, w.T, w.k_lo, d.t_start)
        with pytest.raises(lib.FstatError, match=f"EINVAL.*non-finite SFT bin at {i}$"):
            lib.fstat_set_sfts(*args, x.view(np.complex64)[..., 0])
        with pytest.raises(lib.FstatError, match="EINVAL.*non-finite SFT bin in device input"):
            lib.fstat_set_sfts(*args, torch.from_numpy(x).cuda())
        g.compute()
        np.testing.assert_array_equal(g.twoF(), before)
    finally:
        g.close()
