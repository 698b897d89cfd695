"""The counters of a query do not depend on the batch it comes in: small batches
(which several warps per query, or a CTA per scanned query, would answer) count
what the large batch counts, again and again; and the answers with and without
counters are the same."""
import numpy as np
import pytest

from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")


@pytest.mark.parametrize("storage", [jag.JAG_VEC_F32, jag.JAG_VEC_BF16])
@pytest.mark.parametrize("s0", [0, 4500])
def test_counters_of_parts_are_those_of_the_batch(storage, s0):
    w = D.make_range_i32(n=20000, d=48, nq=1500, seed=91, width=100)
    idx = jag.Index.from_workload(w, R=32, l_b=32, storage=storage)
    f = w.filters.copy()
    lo = np.arange(len(f)) % 400      # sets of 2,000 to 10,000 points: some scanned with s0 = 4,500
    f[:] = D.filters_range_i32(lo, lo + 100 + lo)
    q = torch.from_numpy(w.q).cuda()
    k = 100 if s0 else 10             # of 100 answers the two selections' thresholds differ
    kw = dict(s0=s0, scan_cap=4500, hash_bits=10)
    ids, dist, cnt = idx.search(q, f, w.aux, k, 128, counters=True, **kw)
    assert (cnt[:, 3] == 1).any() == (s0 > 0) and (cnt[:, 3] == 0).any()
    for a, b in ((0, 1), (1, 100), (100, 700), (700, 1500)):
        for _ in range(2):
            pi, pd, pc = idx.search(q[a:b].contiguous(), f[a:b], w.aux, k, 128, counters=True, **kw)
            assert torch.equal(pc, cnt[a:b])
        ni, nd, _ = idx.search(q[a:b].contiguous(), f[a:b], w.aux, k, 128, **kw)
        for i, d in ((pi, pd), (ni, nd)):
            assert torch.equal(i, ids[a:b]) and torch.equal(d, dist[a:b])
    idx.close()
