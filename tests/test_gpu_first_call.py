"""The first call of a process pays for loading the kernels it launches, once each; it must not also
pay for expanding compressed device code, which took ten times as long as the load."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import time
import emd_synth
import paper_1812_02091_gb300 as emd
w = emd_synth.small_text(5, V=600, m=48, n=300, n_queries=2, lo=5, hi=45)
q = w.queries
db = emd.emd_db_create(w.emb, None, w.db.row_ptr, w.db.col, w.db.val,
                       emd.emd_db_options_default(max_query_h=64, autotune=0, graphs=0), v=w.v)
times = []
for _ in range(3):
    t = time.perf_counter()
    emd.emd_topk(db, q.row_ptr, q.col, q.val, "act", 4, "max", 16)
    times.append(time.perf_counter() - t)
emd.emd_db_destroy(db)
print(1e3 * (times[0] - min(times)))
"""


def test_first_search():
    # about a dozen kernels, well below a millisecond each; expanding the reverse pass alone took 10 ms
    extra = []
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr
        extra.append(float(r.stdout.split()[-1]))
    assert min(extra) < 8.0, extra
