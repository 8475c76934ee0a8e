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
