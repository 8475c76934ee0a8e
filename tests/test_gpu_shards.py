"""A divided search against the whole: bit for bit with the forms whose results do not
depend on the sky list, to rounding with the tensor-core form of AUTO."""
import dataclasses

import numpy as np
import pytest

from oracle import fstat_oracle as O
from paper_0904_1826_gb300.multi import shard_range
from tests.test_gpu_tensor import _dense

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_sky,sizes", [(1201, dict(n_sft=11, n_f=301, n_fdot=5, n_bins=340)),
                                         (6000, dict(n_sft=7, n_f=380, n_fdot=1, n_bins=400))])
@pytest.mark.parametrize("algo", ["auto", "sincpoly", "direct"])
def test_shards_against_the_whole_bank(lib, n_sky, sizes, algo):
    """AUTO: both sides within the form's 7e-7 of the exact 2F, so rms 5e-6 apart at most."""
    w = _dense(n_sky, **sizes)
    bins = O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)
    out = []
    for world in (1, 2):
        parts = []
        for rank in range(world):
            lo, hi = shard_range(n_sky, rank, world)
            shard = dataclasses.replace(w, bank=dataclasses.replace(w.bank, sky=w.bank.sky[lo:hi]))
            g = lib.FStat(0, dterms=8, topk=20, algo=algo)
            try:
                g.load_workload(shard, bins_override=bins)
                g.compute()
                assert (g.tensor_tiles()["rows"] > 0) == (algo == "auto") and g.error_flags() == 0
                parts.append(g.twoF())
            finally:
                g.close()
        out.append(np.concatenate(parts))
    if algo == "auto":
        d = out[0].astype(np.float64) - out[1]
        assert np.sqrt(np.mean(d ** 2) / np.mean(out[0].astype(np.float64) ** 2)) <= 5e-6
    else:
        np.testing.assert_array_equal(out[0], out[1])
