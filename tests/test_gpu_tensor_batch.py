"""Batches that hold workunits of the tensor-core form beside others."""
import numpy as np
import pytest

from tests.test_gpu_tensor import ABS, REL, _dense
from workload import config_mid

pytestmark = pytest.mark.gpu

TENSOR = dict(n_sft=11, n_f=301, n_fdot=5, n_bins=340)


def _alone(lib, w):
    g = lib.FStat(0, topk=20)
    try:
        g.load_workload(w)
        g.compute()
        return g.twoF(), g.tensor_tiles()["rows"]
    finally:
        g.close()


def test_batch_autotune_tunes_a_workunit_that_has_tiles(lib):
    """The largest workunit runs on the tensor cores, which have no tiles to tune: the
    largest of the others is timed (stage counts tried: 4, 6, 8; the tensor workunit's
    plan has 3), its M goes to them, and the tensor workunit keeps its plan."""
    wus = [_dense(600, **TENSOR), config_mid(n_sky=40, n_f=150, n_fdot=3), config_mid(n_sky=4, n_f=90, n_fdot=3)]
    alone = [_alone(lib, w) for w in wus]
    assert [rows > 0 for _, rows in alone] == [True, False, False]
    g = lib.FStat(0, topk=20)
    try:
        for w in wus:
            lib.fstat_batch_add(g.ctx, w)
        before = lib.fstat_batch_get_plan(g.ctx, 0)
        t = g.autotune()
        assert t["sft_chunk"] in (4, 6, 8) and t["M"] in (5, 7, 9) and t["slice_us"] > 0
        assert lib.fstat_batch_get_plan(g.ctx, 0) == before
        assert [lib.fstat_batch_get_plan(g.ctx, i)["M"] for i in (1, 2)] == [t["M"]] * 2
        lib.fstat_batch_compute(g.ctx)
        got = [lib.fstat_batch_get_2f(g.ctx, i, 0, w.n_templates) for i, w in enumerate(wus)]
    finally:
        g.close()
    np.testing.assert_array_equal(got[0], alone[0][0])
    for i in (1, 2):
        assert np.all(np.abs(got[i].astype(np.float64) - alone[i][0]) <= 2 * (REL * alone[i][0] + ABS))


def test_batch_autotune_of_tensor_workunits_only_changes_nothing(lib):
    wus = [_dense(600, **TENSOR), _dense(3150, n_sft=4, n_f=193, n_fdot=3, n_bins=230)]
    alone = [_alone(lib, w) for w in wus]
    assert all(rows > 0 for _, rows in alone)
    g = lib.FStat(0, topk=20)
    try:
        for w in wus:
            lib.fstat_batch_add(g.ctx, w)
        before = [lib.fstat_batch_get_plan(g.ctx, i) for i in (0, 1)]
        assert g.autotune()["slice_us"] > 0
        assert [lib.fstat_batch_get_plan(g.ctx, i) for i in (0, 1)] == before
        lib.fstat_batch_compute(g.ctx)
        for i, w in enumerate(wus):
            np.testing.assert_array_equal(lib.fstat_batch_get_2f(g.ctx, i, 0, w.n_templates), alone[i][0])
    finally:
        g.close()


def test_loud_fine_grid_workunit_alone_and_batched(lib):
    """A fine-grid workunit whose bins keep it off the tensor cores falls back to a form
    with a persistent kernel, the same alone and in the batch; a quiet one does not."""
    w = _dense(903, n_sft=8, n_f=511, n_fdot=1, n_bins=120, df_bins=0.125)
    quiet = [d.bins for d in w.detectors]
    loud = [b.copy() for b in quiet]
    loud[0][:, 60] += np.complex64(1e9)
    g = lib.FStat(0, topk=20)
    try:
        for bins in (loud, quiet):
            lib.fstat_batch_add(g.ctx, w, bins)
        one = []
        for i in (0, 1):
            lib.fstat_batch_compute_one(g.ctx, i)
            one.append(lib.fstat_batch_get_2f(g.ctx, i, 0, w.n_templates))
        for _ in range(2):
            lib.fstat_batch_compute(g.ctx)
            for i in (0, 1):
                np.testing.assert_array_equal(lib.fstat_batch_get_2f(g.ctx, i, 0, w.n_templates), one[i])
    finally:
        g.close()
    np.testing.assert_array_equal(one[1], _alone(lib, w)[0])


def test_tensor_workunits_share_one_scratch(lib):
    """Device memory of a batch: a tensor workunit more costs its own tables and 2F, not
    another scratch area (59.8 MB on 152 SMs; the tables and 2F here take 15 MB)."""
    import torch
    w = _dense(600, **TENSOR)
    ref, rows = _alone(lib, w)
    assert rows > 0
    used = []
    for n in (2, 6):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        g = lib.FStat(0, topk=20)
        try:
            for _ in range(n):
                lib.fstat_batch_add(g.ctx, w)
            for _ in range(2):
                lib.fstat_batch_compute(g.ctx)
            for i in range(n):
                np.testing.assert_array_equal(lib.fstat_batch_get_2f(g.ctx, i, 0, w.n_templates), ref)
            used.append(free - torch.cuda.mem_get_info()[0])
        finally:
            g.close()
    assert used[1] - used[0] < 4 * 40e6, used
