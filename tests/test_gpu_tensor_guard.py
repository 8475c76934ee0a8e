"""Guards of the tensor-core form beside tests/test_gpu_tensor.py: its precision (not
only the library's tolerance), noise weights against FP64, SFTs of zeros and of tiny
values, and which kernel runs at full size.

The rms bound, 5e-6 of the rms 2F, is the form's 7e-7 with margin for few SFTs; losing
an FP16 part of the bins or of the weights costs 2^-12 = 2.4e-4.
"""
import dataclasses

import numpy as np
import pytest

from oracle import fstat_oracle as O
from oracle import noise_oracle as N
from tests.test_gpu_fullsize import _read_golden
from tests.test_gpu_tensor import ABS, CASES, REL, _dense
from workload import DetectorData, config1

pytestmark = pytest.mark.gpu

RMS = 5e-6


def _run(lib, w, bins, noise=0, **opts):
    g = lib.FStat(0, dterms=8, topk=20, **opts)
    try:
        g.load_workload(w, bins_override=bins)
        lib.fstat_set_noise_floor(g.ctx, noise)
        g.compute()
        assert g.error_flags() == 0
        return g.twoF().reshape(w.bank.n_sky, w.bank.n_fdot, w.bank.n_f), g.tensor_tiles()["rows"]
    finally:
        g.close()


def _check(got, w, dets):
    pick = sorted({0, w.bank.n_sky // 3, w.bank.n_sky // 2, w.bank.n_sky - 1})
    ref = O.compute_fstat_freq_band(dets, w.T, w.k_lo, 8, dataclasses.replace(w.bank, sky=w.bank.sky[pick]))
    err = got[pick].astype(np.float64) - np.asarray(ref).reshape(len(pick), w.bank.n_fdot, w.bank.n_f)
    assert np.all(np.abs(err) <= REL * np.abs(ref).reshape(err.shape) + ABS)
    assert np.sqrt(np.mean(err ** 2) / np.mean(np.asarray(ref) ** 2)) <= RMS


def _dets(w, bins):
    return [DetectorData(d.lat, d.lon, d.az, d.t_start, b) for d, b in zip(w.detectors, bins)]


@pytest.mark.parametrize("name", [n for n, c in CASES.items() if not c[2]])
@pytest.mark.parametrize("noise", [0, 9])
def test_rms_error_against_fp64(lib, name, noise):
    n_sky, sizes, _, _ = CASES[name]
    w = _dense(n_sky, **sizes)
    bins = O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)
    got, rows = _run(lib, w, bins, noise)
    assert rows > 0
    dets = _dets(w, bins)
    _check(got, w, N.weighted_detectors(dets, noise) if noise else dets)


def test_sfts_of_zeros_and_of_tiny_values(lib):
    """An SFT of zeros (no scale), one 2^-118 as loud (the largest power of two the
    tables take) and data 2^-40 as loud in all (2F exactly 2^-80 as large)."""
    w = _dense(600, n_sft=11, n_f=301, n_fdot=5, n_bins=340)
    bins = O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)
    bins[0][3] = 0
    ordinary = [b.copy() for b in bins]
    bins[1][7] *= np.float32(2.0 ** -118)
    got, rows = _run(lib, w, bins)
    assert rows > 0
    _check(got, w, _dets(w, bins))
    got, _ = _run(lib, w, ordinary)
    small, rows = _run(lib, w, [b * np.float32(2.0 ** -40) for b in ordinary])
    assert rows > 0
    np.testing.assert_array_equal(small, got * np.float32(2.0 ** -80))


@pytest.fixture(scope="module")
def full():
    w = config1()
    return w, O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)


@pytest.mark.parametrize("algo", ["auto", "sincpoly"])
def test_full_size_form_and_parity(lib, full, algo):
    """The whole workunit: AUTO takes the tensor-core form, SINCPOLY the ring with plan
    112 that it replaces.  Each against the oracle's kept top list and every sky point's
    maximum."""
    w, bins = full
    _, g_idx, g_val, sky_max = _read_golden()
    g = lib.FStat(0, topk=w.topk, algo=algo)
    try:
        g.load_workload(w, bins_override=bins)
        g.compute()
        assert g.error_flags() == 0
        assert (g.tensor_tiles()["rows"] > 0) == (algo == "auto") and g.plan()["variant"] == 112
        v = g.twoF()
    finally:
        g.close()
    assert np.all(np.abs(v[g_idx].astype(np.float64) - g_val) <= REL * g_val + ABS)
    top = v.reshape(w.bank.n_sky, -1).max(axis=1)
    assert np.all(np.abs(top.astype(np.float64) - sky_max) <= REL * sky_max + ABS)
