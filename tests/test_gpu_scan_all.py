"""SCAN_ALL on the tensor cores (jag_search) against the brute-force kernels
(jag_search_noalloc): bit-identical answers for every filter kind in one
batch, over more than one group of queries, with and without attribute
columns, at the edges of k; and the CTA-per-query selection of the routed scan
against the warp-per-query one."""
import numpy as np
import pytest

from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")


def _batch(rng, n, d, nq):
    x = (rng.standard_normal((n, d)) + 4 * rng.integers(0, 3, (n, 1))).astype(np.float32)
    q = x[rng.integers(0, n, nq)] + 0.3 * rng.standard_normal((nq, d)).astype(np.float32)
    col = dict(attr_i32=rng.integers(0, 50, n).astype(np.int32), attr_f32=rng.random(n, dtype=np.float32),
               attr_mask=rng.integers(0, 1 << 20, n).astype(np.uint64))
    kind = rng.integers(0, 6, nq)
    f = D.filters_none(nq)
    fb, aux = D.random_bool_filters(rng, nq, 20, 5)
    lo = rng.random(nq).astype(np.float32)
    li = rng.integers(0, 50, nq)
    srcs = {1: D.filters_label(li), 2: D.filters_range_i32(li, li + rng.integers(-1, 9, nq)),   # some empty
            3: D.filters_range_f32(lo, lo + rng.choice([1e-4, 0.05, 1.0], nq).astype(np.float32)),
            4: D.filters_subset(rng.integers(0, 1 << 20, nq) & rng.integers(0, 1 << 20, nq) & rng.integers(0, 1 << 20, nq)),
            5: fb}
    for kd, src in srcs.items():
        f[kind == kd] = src[kind == kd]
    return x, np.ascontiguousarray(q), col, f, aux


def _noalloc(idx, q, f, aux, k):
    ids = torch.empty((len(q), k), dtype=torch.int32, device="cuda")
    dist = torch.empty((len(q), k), dtype=torch.float32, device="cuda")
    jag.jag_search_noalloc(idx.h, q, jag.filters_to_device(f, "cuda"), jag.aux_to_device(aux, "cuda"), k, k, ids, dist,
                           flags=jag.JAG_SEARCH_SCAN_ALL)
    return ids, dist


@pytest.mark.parametrize("n,d,nq,k", [(300_001, 20, 1000, 10), (9_000, 128, 300, 1), (9_000, 300, 70, 128),
                                      (3_000, 33, 40, 129), (130, 8, 30, 100), (1, 4, 3, 2)])
def test_scan_all_matches_brute_force(n, d, nq, k):
    x, q, col, f, aux = _batch(np.random.default_rng(n + k), n, d, nq)
    idx = jag.Index(x, R=4, graph=np.full((n, 4), -1, np.int32), **col)
    qt = torch.from_numpy(q).cuda()
    ids, dist, cnt = idx.search(qt, f, aux, k, k, counters=True, flags=jag.JAG_SEARCH_SCAN_ALL)
    for a in range(0, nq, 200):   # what fits the fixed scratch
        rid, rd = _noalloc(idx, qt[a:a + 200].contiguous(), f[a:a + 200], aux, k)
        assert torch.equal(ids[a:a + 200], rid) and torch.equal(dist[a:a + 200], rd)
    assert (cnt[:, 3] == 2).all()
    idx.close()


def test_scan_all_without_columns():
    x, q, _, _, _ = _batch(np.random.default_rng(3), 5000, 40, 50)
    idx = jag.Index(x, R=4, graph=np.full((5000, 4), -1, np.int32))
    qt = torch.from_numpy(q).cuda()
    ids, dist, _ = idx.search(qt, D.filters_none(50), None, 10, 10, flags=jag.JAG_SEARCH_SCAN_ALL)
    rid, rd = _noalloc(idx, qt, D.filters_none(50), None, 10)
    assert torch.equal(ids, rid) and torch.equal(dist, rd)
    idx.close()


@pytest.mark.parametrize("k", [1, 20, 128, 200])
def test_wide_selection_matches_narrow(k):
    n, d = 60_000, 48
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nq = 8 * sms + 50
    x, q, col, f, aux = _batch(np.random.default_rng(k), n, d, nq)
    idx = jag.Index(x, R=4, graph=np.full((n, 4), -1, np.int32), **col)
    qt = torch.from_numpy(q).cuda()
    ids, dist, cnt = idx.search(qt, f, aux, k, k, counters=True, s0=20_000, scan_cap=20_000)
    routed = cnt[:, 3] == 1
    assert routed.sum() > nq // 2
    for a, b in ((0, 3), (3, 700), (700, nq)):
        pid, pd, pc = idx.search(qt[a:b].contiguous(), f[a:b], aux, k, k, counters=True, s0=20_000, scan_cap=20_000)
        r = routed[a:b]
        assert torch.equal(pc[:, 3], cnt[a:b, 3])
        assert torch.equal(pid[r], ids[a:b][r]) and torch.equal(pd[r], dist[a:b][r])
    idx.close()
