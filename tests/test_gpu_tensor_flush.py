"""The tensor-core form's sums move from registers to tensor memory at the same
SFTs whether or not the SFTs there cover a warp's columns."""
import dataclasses

import numpy as np
import pytest

from oracle import coverage_oracle as CO
from oracle import fstat_oracle as O
from tests.test_gpu_tensor import _dense
from workload import DetectorData

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_sky,sizes,sub", [
    (600, dict(n_sft=150, n_f=301, n_fdot=5, n_bins=340), 1),
    (300, dict(n_sft=150, n_f=639, n_fdot=5, n_bins=360, df_bins=0.5), 2),
])
def test_uncovered_steps_keep_the_sums_order(lib, n_sky, sizes, sub):
    """SFTs (a third of them, 110 of those in a row) that cover nothing of the first 32
    columns, whose warps skip them, against the same SFTs covering the last template of
    those columns too, whose warps mask them: the other templates there get the same
    terms, so the same 2F to the last bit.  And within 5e-6 (rms) of FP64: the form's
    7e-7 with margin, as for all its sums."""
    w = _dense(n_sky, **sizes)
    bins = O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)
    n, nf = w.n_sft_total, w.bank.n_f
    off = np.random.default_rng(8).random(n) < 0.3
    off[120:230] = True
    first = 32 * sub
    out = []
    for edge in (first, first - 1):
        lo = np.where(off, edge, 0).astype(np.int32)
        g = lib.FStat(0, dterms=8, topk=20)
        try:
            g.load_workload(w, bins_override=bins)
            lib.fstat_set_coverage(g.ctx, lo, np.full(n, nf, np.int32))
            g.compute()
            assert g.tensor_tiles()["rows"] > 0
            out.append(g.twoF().reshape(w.bank.n_sky, w.bank.n_fdot, nf))
        finally:
            g.close()
    np.testing.assert_array_equal(out[0][..., :first - 1], out[1][..., :first - 1])
    pick = [0, n_sky // 3, n_sky - 1]
    dets = [DetectorData(d.lat, d.lon, d.az, d.t_start, b) for d, b in zip(w.detectors, bins)]
    part = dataclasses.replace(w.bank, sky=w.bank.sky[pick], n_f=first)
    lo = np.where(off, first, 0).astype(np.int32)
    ref = CO.compute_fstat_coverage(dets, w.T, w.k_lo, 8, part, lo, np.full(n, nf, np.int32)).reshape(3, -1, first)
    err = out[0][pick][..., :first] - ref
    assert np.sqrt(np.mean(err ** 2) / np.mean(ref ** 2)) <= 5e-6
