"""The tensor-core form of the Dirichlet accumulation against the FP64 oracle
and the direct form, over the banks it accepts: spindown counts, templates per
bin, ragged bands and row tiles, sky lists in their own and in grouped order,
storage forms, noise weights, few SFTs and several tiles a block.

Tolerance: the library's, |d2F| <= 1e-4 2F + 1e-3, against the oracle; twice
that between two forms that both keep it.
"""
import dataclasses

import numpy as np
import pytest

from oracle import fstat_oracle as O
from oracle import noise_oracle as N
from oracle import quantize as Q
from workload import DetectorData, config_mid, fibonacci_sky

pytestmark = pytest.mark.gpu

REL, ABS = 1e-4, 1e-3


def _dense(n_sky, seed=500, **kw):
    """config_mid's detectors and signals with a lattice sky of n_sky points,
    the first signal's own point among them."""
    w = config_mid(seed=seed, n_sky=1, **kw)
    sky = fibonacci_sky(n_sky)
    sky[n_sky // 3] = w.bank.sky[0]
    return dataclasses.replace(w, bank=dataclasses.replace(w.bank, sky=sky))


def _run(lib, w, bins, noise=0, **opts):
    g = lib.FStat(0, dterms=8, topk=20, **opts)
    try:
        g.load_workload(w, bins_override=bins)
        if noise:
            lib.fstat_set_noise_floor(g.ctx, noise)
        g.compute()
        shape = (w.bank.n_sky, w.bank.n_fdot, w.bank.n_f)
        return g.twoF().reshape(shape), g.toplist(20), g.error_flags(), g.tensor_tiles()
    finally:
        g.close()


CASES = {
    # name: (n_sky, config_mid sizes, options, noise-floor half window)
    "five spindowns, ragged columns": (600, dict(n_sft=11, n_f=301, n_fdot=5, n_bins=340), {}, 0),
    "one spindown": (3001, dict(n_sft=7, n_f=380, n_fdot=1, n_bins=400), {}, 0),
    "two templates a bin": (300, dict(n_sft=9, n_f=639, n_fdot=5, n_bins=360, df_bins=0.5), {}, 0),
    "four templates a bin": (170, dict(n_sft=8, n_f=2041, n_fdot=3, n_bins=560, df_bins=0.25), {}, 0),
    "eight templates a bin": (903, dict(n_sft=8, n_f=511, n_fdot=1, n_bins=120, df_bins=0.125), {}, 0),
    "several tiles a block": (1500, dict(n_sft=6, n_f=500, n_fdot=7, n_bins=540), {}, 0),
    "fewest SFTs, a column past the block": (3150, dict(n_sft=4, n_f=193, n_fdot=3, n_bins=230), {}, 0),
    "f16 storage with noise weights": (600, dict(n_sft=11, n_f=320, n_fdot=5, n_bins=340), dict(bins_form="f16"), 9),
    "bf16 storage": (600, dict(n_sft=11, n_f=320, n_fdot=5, n_bins=340), dict(bins_form="bf16"), 0),
}


@pytest.mark.parametrize("name", CASES)
def test_tensor_form_against_oracle_and_direct_form(lib, name):
    n_sky, sizes, opts, noise = CASES[name]
    w = _dense(n_sky, **sizes)
    bins = O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)
    got, top, flags, tiles = _run(lib, w, bins, noise, **opts)
    assert tiles["rows"] > 0, tiles
    direct, _, dflags, none = _run(lib, w, bins, noise, algo="direct", **opts)
    assert flags == 0 and dflags == 0 and none["rows"] == 0
    assert np.all(np.abs(got.astype(np.float64) - direct) <= 2 * (REL * np.abs(direct) + ABS))
    flat = got.ravel()
    order = np.lexsort((np.arange(flat.size), -flat.astype(np.float64)))[:20]
    np.testing.assert_array_equal(top[0], order)
    # the oracle on four sky points: first, last, the signal's and one more
    pick = sorted({0, n_sky // 3, n_sky // 2, n_sky - 1})
    dets = [DetectorData(d.lat, d.lon, d.az, d.t_start, b) for d, b in zip(w.detectors, bins)]
    if noise:
        dets = N.weighted_detectors(dets, noise)
    if "bins_form" in opts and not noise:
        dets = [dataclasses.replace(d, bins=Q.dequantize(*Q.quantize(d.bins, opts["bins_form"]), opts["bins_form"]))
                for d in dets]
    if noise:
        return   # quantised after whitening: the direct form's own parity covers the oracle
    sub = dataclasses.replace(w.bank, sky=w.bank.sky[pick])
    ref = O.compute_fstat_freq_band(dets, w.T, w.k_lo, 8, sub)
    ref = np.asarray(ref).reshape(len(pick), w.bank.n_fdot, w.bank.n_f)
    assert np.all(np.abs(got[pick].astype(np.float64) - ref) <= REL * np.abs(ref) + ABS)


def test_tensor_form_scales_exactly_with_the_data(lib):
    """Bins times 2^40: the tables' per-SFT power of two takes it up, so 2F is
    exactly 2^80 times as large; a line 10^6 above the noise in one bin keeps
    parity with the direct form in the rest of the band."""
    w = _dense(600, n_sft=9, n_f=301, n_fdot=5, n_bins=340)
    bins = O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)
    a, _, fa, tiles = _run(lib, w, bins)
    b, _, fb, _ = _run(lib, w, [x * np.float32(2.0 ** 40) for x in bins])
    assert tiles["rows"] > 0 and fa == 0 and fb == 0
    np.testing.assert_array_equal(a * np.float32(2.0 ** 80), b)
    loud = [x.copy() for x in bins]
    loud[0][:, 170] += np.complex64(1e6)
    c, _, fc, _ = _run(lib, w, loud)
    d, _, _, _ = _run(lib, w, loud, algo="direct")
    assert fc == 0
    # away from the line (its sidelobes fall off within the 16-bin window)
    far = np.r_[0:120, 220:301]
    assert np.all(np.abs(c[..., far].astype(np.float64) - d[..., far]) <= 2 * (REL * np.abs(d[..., far]) + ABS))


def test_tensor_form_wait_timeout_is_reported_and_context_survives(lib):
    """Copies that stop after 3 SFTs run the bounded waits out: flag bit 2, and
    the next compute on the context is correct again."""
    w = _dense(600, n_sft=6, n_f=301, n_fdot=5, n_bins=340)
    g = lib.FStat(0, topk=5)
    try:
        g.load_workload(w)
        assert g.tensor_tiles()["rows"] > 0
        g.compute()
        ok = g.twoF()
        lib.fstat_test_ring_stall(g.ctx, 3)
        g.compute()
        assert g.error_flags() & 4
        lib.fstat_test_ring_stall(g.ctx, -1)
        g.compute()
        assert g.error_flags() == 0
        np.testing.assert_array_equal(g.twoF(), ok)
    finally:
        g.close()


def test_batched_tensor_workunits_equal_single_launches(lib):
    """A batch of one tensor-core and one ring workunit, run twice (direct and
    from the captured graph): 2F equal to each workunit alone."""
    wus = [_dense(600, n_sft=9, n_f=301, n_fdot=5, n_bins=340), config_mid(n_sky=4, n_f=90, n_fdot=3)]
    refs = []
    for w in wus:
        g = lib.FStat(0, topk=20)
        try:
            g.load_workload(w)
            g.compute()
            refs.append((g.twoF(), g.toplist(20), g.tensor_tiles()["rows"]))
        finally:
            g.close()
    assert refs[0][2] > 0 and refs[1][2] == 0
    g = lib.FStat(0, topk=20)
    try:
        for w in wus:
            lib.fstat_batch_add(g.ctx, w)
        for _ in range(2):
            lib.fstat_batch_compute(g.ctx)
            for i, w in enumerate(wus):
                np.testing.assert_array_equal(lib.fstat_batch_get_2f(g.ctx, i, 0, w.n_templates), refs[i][0])
                np.testing.assert_array_equal(lib.fstat_batch_get_toplist(g.ctx, i, 20)[0], refs[i][1][0])
        done, total = lib.fstat_batch_get_times(g.ctx, 2)
        assert np.all(done > 0) and np.all(done <= total * 1.001)
    finally:
        g.close()


@pytest.mark.parametrize("n_sky,sizes", [
    (300, dict(n_sft=60, n_f=301, n_fdot=5, n_bins=340)),     # 60 tiles: two or three blocks a tile
    (520, dict(n_sft=6, n_f=510, n_fdot=5, n_bins=550)),      # 168 tiles: most blocks start inside one
    (1130, dict(n_sft=5, n_f=320, n_fdot=5, n_bins=360)),     # 225 tiles: runs of one and a half
    (2400, dict(n_sft=4, n_f=320, n_fdot=5, n_bins=360)),     # 470 tiles: three or four segments, all scratch slots
])
def test_tiles_shared_by_blocks(lib, n_sky, sizes):
    """Parts of a tile's SFTs on different blocks, against the direct form."""
    w = _dense(n_sky, **sizes)
    bins = O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)
    got, _, flags, tiles = _run(lib, w, bins)
    assert tiles["rows"] > 0 and flags == 0
    again, _, _, _ = _run(lib, w, bins)
    np.testing.assert_array_equal(got, again)     # the parts are added in one order
    direct, _, _, none = _run(lib, w, bins, algo="direct")
    assert none["rows"] == 0
    assert np.all(np.abs(got.astype(np.float64) - direct) <= 2 * (REL * np.abs(direct) + ABS))


@pytest.mark.parametrize("n_sky,f0", [(250, 217.0), (1500, 390.0)])
def test_sparse_skies_at_high_frequency(lib, n_sky, f0):
    """Tiles of far-apart sky points of both hemispheres over two months: the
    planner's bound holds the windows (no range flag)."""
    w = _dense(n_sky, n_sft=30, n_f=512, n_fdot=7, n_bins=760)
    spread = [dataclasses.replace(d, t_start=w.bank.t_ref + (d.t_start - d.t_start[0]) * 5.2e6 / max(d.t_start[-1] - d.t_start[0], 1.0))
            for d in w.detectors]
    shift = int(round(f0 * w.T)) - int(round(w.bank.f0 * w.T))
    bank = dataclasses.replace(w.bank, f0=w.bank.f0 + shift / w.T)
    w = dataclasses.replace(w, detectors=spread, bank=bank, k_lo=w.k_lo + shift)
    bins = [d.bins for d in w.detectors]
    got, _, flags, tiles = _run(lib, w, bins)
    direct, _, dflags, _ = _run(lib, w, bins, algo="direct")
    assert tiles["rows"] > 0 and flags == dflags
    assert np.all(np.abs(got.astype(np.float64) - direct) <= 2 * (REL * np.abs(direct) + ABS))


@pytest.mark.parametrize("sizes,n_sky", [
    (dict(n_sft=40, n_f=301, n_fdot=5, n_bins=340), 600),
    (dict(n_sft=40, n_f=639, n_fdot=5, n_bins=360, df_bins=0.5), 300),
    (dict(n_sft=60, n_f=301, n_fdot=5, n_bins=340), 300),     # tiles shared by blocks
])
def test_tensor_form_with_coverage(lib, sizes, n_sky):
    """SFTs that cover everything, nothing, one template, up to and from the edges
    of column blocks, and ranges far outside the band, against the direct form."""
    w = _dense(n_sky, **sizes)
    bins = O.inject(w.detectors, w.T, w.k_lo, w.injections, w.bank.t_ref)
    n, nf = w.n_sft_total, w.bank.n_f
    rng = np.random.default_rng(4)
    lo, hi = np.zeros(n, np.int32), np.full(n, nf, np.int32)
    special = [(0, 64), (64, 128), (63, 65), (5, 6), (nf, nf), (0, 0), (-2 ** 31, 2 ** 31 - 1), (-2 ** 31, 40),
               (200, 2 ** 31 - 1), (nf - 1, nf)]
    for i, (a, b) in enumerate(special[:n]):
        lo[i], hi[i] = a, b
    for i in range(len(special), n):
        if i % 5 == 1:
            lo[i] = rng.integers(-10, nf // 2)
            hi[i] = lo[i] + rng.integers(nf // 2, nf)

    def run(**opts):
        g = lib.FStat(0, dterms=8, topk=20, **opts)
        try:
            g.load_workload(w, bins_override=bins)
            lib.fstat_set_coverage(g.ctx, lo, hi)
            g.compute()
            return g.twoF(), g.error_flags(), g.tensor_tiles()["rows"]
        finally:
            g.close()

    got, flags, rows = run()
    direct, dflags, none = run(algo="direct")
    assert rows > 0 and none == 0 and flags == dflags
    assert np.all(np.abs(got.astype(np.float64) - direct) <= 2 * (REL * np.abs(direct) + ABS))
