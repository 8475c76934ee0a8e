"""Strong lines and the tensor-core form: its tables scale an SFT by one power of
two, so beside a line far above the noise the planner keeps a form with FP32 bins.

Bounds: the library's, |d2F| <= 1e-4 2F + 1e-3, and 5e-6 for the rms error over the
rms 2F.  Both forms' sums carry 7e-7 (tensor) to 2e-6 (sinc polynomial); the rest is
margin for the few SFTs here.  A line of 10^8 in the tables would cost 1.8e-4 of Fa
and Fb.
"""
import dataclasses

import numpy as np
import pytest

from oracle import fstat_oracle as O
from tests.test_gpu_tensor import ABS, REL, _dense
from workload import DetectorData

pytestmark = pytest.mark.gpu

RMS = 5e-6


def _context(lib, w, bins, **opts):
    g = lib.FStat(0, dterms=8, topk=20, **opts)
    g.load_workload(w, bins_override=bins)
    return g


def _check(got, w, bins, cols):
    """2F [n_sky, n_fdot, n_f] at four sky points and the columns `cols` against the oracle."""
    pick = sorted({0, w.bank.n_sky // 3, w.bank.n_sky // 2, w.bank.n_sky - 1})
    dets = [DetectorData(d.lat, d.lon, d.az, d.t_start, b) for d, b in zip(w.detectors, bins)]
    ref = O.compute_fstat_freq_band(dets, w.T, w.k_lo, 8, dataclasses.replace(w.bank, sky=w.bank.sky[pick]))
    ref = np.asarray(ref).reshape(len(pick), w.bank.n_fdot, w.bank.n_f)[..., cols]
    err = got[pick][..., cols].astype(np.float64) - ref
    assert np.all(np.abs(err) <= REL * np.abs(ref) + ABS)
    assert np.sqrt(np.mean(err ** 2) / np.mean(ref ** 2)) <= RMS


def _shape(w):
    return w.bank.n_sky, w.bank.n_fdot, w.bank.n_f


@pytest.mark.parametrize("line,tensor", [(0.0, True), (1e3, True), (3e4, True), (1e7, False), (1e8, False), (1e9, False),
                                         (1e10, False)])
def test_templates_away_from_a_line(lib, line, tensor):
    w = _dense(600, n_sft=11, n_f=301, n_fdot=5, n_bins=340)
    bins = O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)
    bins[0][:, 170] += np.complex64(line)
    g = _context(lib, w, bins)
    try:
        g.compute()
        got, flags, rows = g.twoF().reshape(_shape(w)), g.error_flags(), g.tensor_tiles()["rows"]
    finally:
        g.close()
    assert flags == 0 and (rows > 0) == tensor
    # the line's window and the Doppler shift (18 bins) stay out
    _check(got, w, bins, np.r_[0:120, 220:301] if line else np.r_[0:301])


@pytest.mark.parametrize("form,line", [("bf16", 1e9), ("c64", 1e10)])
def test_line_outside_the_banks_windows(lib, form, line):
    """A narrow bank in a wide band: a line that no window reaches changes nothing."""
    w = _dense(600, n_sft=11, n_f=301, n_fdot=5, n_bins=1100)
    w = dataclasses.replace(w, bank=dataclasses.replace(w.bank, f0=(w.k_lo + 300) / w.T))
    quiet = [d.bins for d in w.detectors]
    loud = [b.copy() for b in quiet]
    loud[1][:, 800] += np.complex64(line)
    out = []
    for bins in (quiet, loud):
        g = _context(lib, w, bins, bins_form="c64")
        try:
            g.compute()
            assert g.tensor_tiles()["rows"] > 0 and g.error_flags() == 0
            out.append(g.twoF().reshape(_shape(w)))
        finally:
            g.close()
    np.testing.assert_array_equal(out[0], out[1])
    _check(out[1], w, loud, np.r_[0:301])
    # the same line inside the windows, in the storage form: another form runs
    loud[1][:, 450] += np.complex64(line)
    g = _context(lib, w, loud, bins_form=form)
    try:
        assert g.tensor_tiles()["rows"] == 0
    finally:
        g.close()


def test_form_follows_the_bins_under_one_bank(lib):
    """Bins replaced or whitened under an unchanged bank: the form follows.  A signal
    alone, however loud, leaves no quiet window: its sidelobes fall off as 1 / (pi d)
    over the 340 bins."""
    w = _dense(600, n_sft=11, n_f=301, n_fdot=5, n_bins=340)
    quiet = [d.bins for d in w.detectors]
    sig = dataclasses.replace(w.injections[0], rho=1e12)
    g = _context(lib, w, quiet)
    try:
        g.compute()
        assert g.tensor_tiles()["rows"] > 0
        first = g.twoF()
        lib.fstat_inject(g.ctx, [sig], w.bank.t_ref)
        g.compute()
        assert g.tensor_tiles()["rows"] > 0 and g.error_flags() == 0
        bins = [lib.fstat_get_bins(g.ctx, i, d.n_sft, w.n_bins) for i, d in enumerate(w.detectors)]
        _check(g.twoF().reshape(_shape(w)), w, bins, np.r_[0:301])
        for i, x in enumerate(w.detectors):
            lib.fstat_set_sfts(g.ctx, i, x.lat, x.lon, x.az, w.T, w.k_lo, x.t_start, quiet[i])
        g.compute()
        assert g.tensor_tiles()["rows"] > 0
        np.testing.assert_array_equal(g.twoF(), first)
        # half the band 10^6 louder: whitened, it is level again
        step = [b * np.where(np.arange(b.shape[1]) < 170, 1e6, 1.0).astype(np.float32) for b in quiet]
        for i, x in enumerate(w.detectors):
            lib.fstat_set_sfts(g.ctx, i, x.lat, x.lon, x.az, w.T, w.k_lo, x.t_start, step[i])
        assert g.tensor_tiles()["rows"] == 0
        lib.fstat_set_noise_floor(g.ctx, 9)
        assert g.tensor_tiles()["rows"] > 0
        g.compute()
        assert g.error_flags() == 0
        lib.fstat_set_noise_floor(g.ctx, 0)
        assert g.tensor_tiles()["rows"] == 0
    finally:
        g.close()


@pytest.mark.parametrize("start,width,tensor", [(400, 16, False), (400, 15, True), (2033 - 15, 16, False), (2033, 15, True),
                                                (2033, 16, False), (2040, 16, False), (2048 - 15, 17, False),
                                                (4081, 16, False), (4081, 15, True), (4900, 16, False)])
def test_quiet_windows_are_found_wherever_they_start(lib, start, width, tensor):
    """16 weak bins in a row in one SFT make a quiet window, 15 do not, across the
    pieces in which the range is scanned."""
    w = _dense(600, n_sft=4, n_f=4900, n_fdot=3, n_bins=5000)
    bins = [d.bins.copy() for d in w.detectors]
    bins[1][2, start:start + width] = np.complex64(1e-6 + 1e-6j)
    g = _context(lib, w, bins)
    try:
        assert (g.tensor_tiles()["rows"] > 0) == tensor
    finally:
        g.close()
