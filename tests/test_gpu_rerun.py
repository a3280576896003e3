"""Queries of the fused form that are not certified run once more with the full distance matrix.
Those sequences rarely come again, so they are launched directly: no graph is captured for them
(a capture costs more than it could save, and in a server it holds up the other executors)."""
import numpy as np
import pytest

import emd_synth

pytestmark = pytest.mark.gpu


def test_reruns_capture_no_graph():
    import paper_1812_02091_gb300 as emd
    w = emd_synth.small_text(21, V=900, m=48, n=400, n_queries=8, lo=3, hi=45, qlo=5, qhi=60)
    db = w.db.subset(np.concatenate([np.arange(400), np.repeat([3, 77], 300)]))  # 300 documents tie at distance 0
    h = emd.emd_db_create(w.emb, None, db.row_ptr, db.col, db.val,
                          emd.emd_db_options_default(precision="fp32_tc", max_query_h=64, autotune=0), v=w.v)
    try:
        calls = 0
        for doc in (3, 77, 3):
            idx, val = w.db.row(doc)
            got, dist = emd.emd_topk(h, np.array([0, len(idx)], np.int64), idx, val, "act", 4, "max", 16)
            calls += 1
            p = emd.emd_db_profile_get(h)
            assert p["prune_fallbacks"] == calls  # the call did rerun its query
            assert p["graph_launches"] == calls   # ... beside its one captured batch
            assert not dist.any()                 # 16 copies of the query
            np.testing.assert_array_equal(got[0], np.flatnonzero([np.array_equal(db.row(i)[0], idx) and
                                                                  np.array_equal(db.row(i)[1], val)
                                                                  for i in range(db.n)])[:16])
    finally:
        emd.emd_db_destroy(h)
