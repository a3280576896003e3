"""The batched forward sweep at the ends of its dispatch, against the per-query pass bit for bit: groups of
16 queries whose tables have one entry (the only ones that come in 16), and databases of more than
200,000 documents, where a warp takes four and its range can cross from the long documents to the
others."""
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


def test_four_documents_per_warp(emd):
    rng = np.random.Generator(np.random.PCG64(6))
    n, n_long = 200005, 37  # 200,042 places: the last warp has two
    w = emd_synth.small_text(42, V=1200, m=40, n=50, n_queries=9, lo=1, hi=40, qlo=1, qhi=40)
    lengths = rng.integers(1, 5, size=n)
    lengths[np.r_[0, n - 1, rng.permutation(np.arange(1, n - 1))[: n_long - 2]]] = rng.integers(33, 300, size=n_long)
    db = emd_synth.zipf_histograms(rng, 1200, lengths)
    _equal(emd, w, db, w.queries, [("rwmd", 1), ("omr", 1), ("act", 1), ("act", 4)], max_query_h=64)
    _equal(emd, w, db, w.queries.subset(range(1)), [("rwmd", 1), ("act", 3)], max_query_h=64)
