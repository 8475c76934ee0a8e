"""bench.py states the 2F error of the kernel that it times."""
import dataclasses

import numpy as np
import pytest

import bench
from oracle import fstat_oracle as O
from tests.test_gpu_tensor import _dense
from workload import DetectorData

pytestmark = pytest.mark.gpu


def test_error_is_taken_from_the_timed_kernel(lib):
    """A sample of sky points, too few for the tensor-core form by themselves, of a bank
    that runs on it."""
    w = _dense(600, n_sft=11, n_f=301, n_fdot=5, n_bins=340)
    bins = O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)
    pick = [0, 200, 599]
    sub = dataclasses.replace(w.bank, sky=w.bank.sky[pick])
    dets = [DetectorData(d.lat, d.lon, d.az, d.t_start, b) for d, b in zip(w.detectors, bins)]
    ref = np.asarray(O.compute_fstat_freq_band(dets, w.T, w.k_lo, 8, sub))
    got = bench.gpu_2f_error(w, pick, bins, sub, ref, 0, None, bins_form="c64", algo="auto")
    assert got["chosen"]["kernel"] == "dirichlet_tc_kernel" and got["plain_fp32"]["kernel"] == "dirichlet_kernel"
    g = lib.FStat(0, dterms=8, topk=10)
    try:
        g.load_workload(w, bins_override=bins)
        g.compute()
        mine = g.twoF().reshape(600, -1)[pick].astype(np.float64)
    finally:
        g.close()
    assert got["chosen"]["max_abs"] == np.abs(mine - ref.reshape(3, -1)).max()
    assert got["chosen"]["max_over_tol"] <= 1.0
