"""The batched forward sweep at the ends of its dispatch, against the per-query pass bit for bit: groups of
16 queries whose tables have one entry (the only ones that come in 16)."""
import numpy as np
import pytest

import emd_synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def emd():
    import paper_1812_02091_gb300 as m
    m.load()
    return m


def _equal(emd, w, db, q, calls, **opt):
    h = [emd.emd_db_create(w.emb, None, db.row_ptr, db.col, db.val,
                           emd.emd_db_options_default(autotune=0, batched=b, **opt), v=w.v) for b in (1, 0)]
    try:
        for meas, k in calls:
            got, want = (emd.emd_query_batch(x, q.row_ptr, q.col, q.val, meas, k, "fwd") for x in h)
            np.testing.assert_array_equal(got, want)
    finally:
        for x in h:
            emd.emd_db_destroy(x)


@pytest.mark.parametrize("nq", [9, 16, 17, 33])
def test_sixteen_one_bin_queries(emd, nq):
    w = emd_synth.small_text(41, V=700, m=40, n=300, n_queries=2, lo=1, hi=40)
    ids = (np.arange(nq) * 19 % 700).astype(np.int32)
    q = emd_synth.Histograms(np.arange(nq + 1, dtype=np.int64), ids, np.ones(nq, np.float32))
    _equal(emd, w, w.db, q, [("rwmd", 1), ("omr", 1), ("act", 4), ("act", 1), ("ict", 1)], max_query_h=1)
