"""jag_search_host through the one-copy staging of small calls and through the
array-by-array copies of larger ones: the answers, counters and errors of the
device-pointer search."""
import numpy as np
import pytest

from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")


@pytest.fixture(scope="module")
def case():
    w = D.make_mixed(n=4000, d=37, nq=1500, seed=80, n_centres=10)
    return w, jag.Index.from_workload(w, R=24, l_b=32)


# 37-d queries with counters and k = 10 take about 300 bytes each: the line lies near 850 queries
@pytest.mark.parametrize("nq", [1, 3, 840, 850, 860, 1500])
def test_host_search_is_the_device_search(case, nq):
    w, idx = case
    ids, dist, cnt = idx.search_host(w.q[:nq], w.filters[:nq], w.aux, 10, 40, counters=True)
    rid, rd, rc = idx.search(torch.from_numpy(w.q[:nq]).cuda(), w.filters[:nq], w.aux, 10, 40, counters=True)
    assert np.array_equal(ids, rid.cpu().numpy()) and np.array_equal(dist, rd.cpu().numpy())
    assert np.array_equal(cnt[:, [0, 3]], rc.cpu().numpy()[:, [0, 3]])


def test_small_call_reports_bad_filters(case):
    w, idx = case
    f = w.filters[:4].copy()
    f["kind"][2] = 77
    ids = np.zeros((4, 10), np.int32)
    with pytest.raises(jag.JagError) as e:
        idx.search_host(w.q[:4], f, w.aux, 10, 40, out_ids=ids)
    assert e.value.status == jag.JAG_EINVAL
    assert (ids[2] == -1).all() and (ids[0] >= 0).any()
