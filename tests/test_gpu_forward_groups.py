"""The batched forward sweep groups 1, 2, 4, 8 or 16 queries by the batch's size and stores
their tables by pairs of entries; every value equals the per-query pass's bit for bit, for
batch sizes on both sides of each group size, odd table widths, documents of one bin up to
several steps of the sweep, and one-bin queries."""
import numpy as np
import pytest

import emd_synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def emd():
    import paper_1812_02091_gb300 as m
    m.load()
    return m


@pytest.fixture(scope="module")
def work():
    w = emd_synth.small_text(31, V=1500, m=40, n=500, n_queries=35, lo=1, hi=40, qlo=1, qhi=70)
    rng = np.random.Generator(np.random.PCG64(5))
    long = emd_synth.zipf_histograms(rng, 1500, np.array([129, 400, 777, 131, 260]))  # past twice the mean length
    rp = np.concatenate([w.db.row_ptr, w.db.row_ptr[-1] + long.row_ptr[1:]])
    return w, emd_synth.Histograms(rp, np.concatenate([w.db.col, long.col]), np.concatenate([w.db.val, long.val]))


@pytest.mark.parametrize("precision", ["fp32", "fp32_tc", "bf16"])
@pytest.mark.parametrize("meas,k", [("rwmd", 1), ("omr", 1), ("act", 1), ("act", 2), ("act", 3), ("act", 4), ("act", 7),
                                    ("act", 16), ("ict", 1)])
def test_groups_equal_per_query(emd, work, precision, meas, k):
    if precision == "bf16" and meas == "ict":
        pytest.skip("ICT re-rank width")
    w, db = work
    h = [emd.emd_db_create(w.emb, None, db.row_ptr, db.col, db.val,
                           emd.emd_db_options_default(precision=precision, max_query_h=128, autotune=0, batched=b), v=w.v)
         for b in (1, 0)]
    try:
        for nq in (1, 2, 3, 4, 5, 8, 9, 17, 35):
            q = w.queries.subset(range(nq))
            got, want = (emd.emd_query_batch(x, q.row_ptr, q.col, q.val, meas, k, "fwd") for x in h)
            np.testing.assert_array_equal(got, want)
    finally:
        for x in h:
            emd.emd_db_destroy(x)


@pytest.mark.parametrize("meas", ["rwmd", "omr", "act", "ict"])
def test_one_bin_queries(emd, work, meas):
    w, db = work
    ids = np.array([0, 3, 700, 1499], np.int32)  # tables of one entry: max_query_h = 1
    h = [emd.emd_db_create(w.emb, None, db.row_ptr, db.col, db.val,
                           emd.emd_db_options_default(max_query_h=1, autotune=0, batched=b), v=w.v) for b in (1, 0)]
    try:
        got, want = (emd.emd_query_batch(x, np.arange(5), ids, np.ones(4, np.float32), meas, 4, "fwd") for x in h)
        np.testing.assert_array_equal(got, want)
    finally:
        for x in h:
            emd.emd_db_destroy(x)
