"""SCAN_ALL on both sides of the lines between the tensor cores and the
brute-force kernel -- few points, boolean and subset filters of large batches,
passing sets too large for the scratch -- with every filter kind in one batch,
against the brute-force kernel alone (jag_search_noalloc)."""
import numpy as np
import pytest

from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")

BITS = 12


def _index(n, d, seed, mask=True):
    rng = np.random.default_rng(seed)
    col = dict(attr_i32=rng.integers(0, 30, n).astype(np.int32), attr_f32=rng.random(n, dtype=np.float32))
    if mask:
        col["attr_mask"] = rng.integers(0, 1 << BITS, n).astype(np.uint64)
    return jag.Index(rng.standard_normal((n, d)).astype(np.float32), R=1, graph=np.full((n, 1), -1, np.int32), **col)


def _filters(nq, seed, mask=True):
    rng = np.random.default_rng(seed)
    f = D.filters_none(nq)
    fb, aux = D.random_bool_filters(rng, nq, BITS, 4)
    lo = rng.random(nq).astype(np.float32)
    li = rng.integers(0, 30, nq)
    srcs = {1: D.filters_label(li), 2: D.filters_range_i32(li, li + rng.integers(-1, 25, nq)),
            3: D.filters_range_f32(lo, lo + rng.choice([1e-3, 0.2, 1.0], nq).astype(np.float32)),
            4: D.filters_subset(rng.integers(0, 1 << BITS, nq) & rng.integers(0, 1 << BITS, nq) & rng.integers(0, 1 << BITS, nq)),
            5: fb}
    kind = np.arange(nq) % (6 if mask else 4)
    for kd, src in srcs.items():
        f[kind == kd] = src[kind == kd]
    return f, aux


def _check(idx, n, d, nq, k, mask=True):
    f, aux = _filters(nq, nq, mask)
    q = torch.from_numpy(np.random.default_rng(n).standard_normal((nq, d)).astype(np.float32)).cuda()
    ids, dist, cnt = idx.search(q, f, aux, k, k, counters=True, flags=jag.JAG_SEARCH_SCAN_ALL)
    assert (cnt.cpu().numpy() == [0, 0, 0, 2]).all()
    ft, at = jag.filters_to_device(f, "cuda").view(-1, 16), jag.aux_to_device(aux, "cuda")
    rid, rd = torch.empty_like(ids), torch.empty_like(dist)
    step = 100   # what fits the fixed scratch
    for a in range(0, nq, step):
        jag.jag_search_noalloc(idx.h, q[a:a + step].contiguous(), ft[a:a + step].contiguous(), at, k, k,
                               rid[a:a + step], rd[a:a + step], flags=jag.JAG_SEARCH_SCAN_ALL)
    assert torch.equal(ids, rid) and torch.equal(dist, rd)


# 2,048 points; boolean filters (a sixth of the queries) on both sides of their lines: n (50 + d) ns against 0.1 ms +
# 12.5 us a filter of the first 64 + n / 50 ns a filter, and 1.2 * 10^8 / n
@pytest.mark.parametrize("n,d,nq", [(2047, 24, 60), (2048, 24, 60), (2100, 64, 126), (2100, 64, 132), (9000, 24, 264),
                                    (9000, 24, 270), (100_001, 24, 7199), (100_001, 24, 7200)])
def test_lines_of_small_indexes(n, d, nq):
    idx = _index(n, d, n)
    _check(idx, n, d, nq, 10)
    idx.close()


def test_lines_of_large_indexes():
    n, d = (1 << 22) + 77, 4
    idx = _index(n, d, 1)
    for nq, k in ((5, 10), (31, 100), (50, 10), (200, 10)):   # all sets kept; those past 2M rows not
        _check(idx, n, d, nq, k)
    idx.close()
    idx = _index(n, d, 2, mask=False)
    for nq in (60, 70, 130):
        _check(idx, n, d, nq, 10, mask=False)
    idx.close()


@pytest.mark.parametrize("d", [48, 300, 600])
@pytest.mark.parametrize("k", [1, 20, 128, 200])
def test_routed_scan_with_and_without_counters(k, d):
    """A CTA per routed query (no counters) against a warp per query."""
    n, nq = 30_000, 600
    idx = _index(n, d, k + d)
    f, aux = _filters(nq, k)
    q = torch.from_numpy(np.random.default_rng(k).standard_normal((nq, d)).astype(np.float32)).cuda()
    kw = dict(s0=20_000, scan_cap=20_000)
    for a, b in ((0, 3), (3, nq)):
        rid, rd, cnt = idx.search(q[a:b].contiguous(), f[a:b], aux, k, k, counters=True, **kw)
        ids, dist, _ = idx.search(q[a:b].contiguous(), f[a:b], aux, k, k, **kw)
        assert b == 3 or (cnt[:, 3] == 1).sum() > nq // 2
        assert torch.equal(ids, rid) and torch.equal(dist, rd)
    idx.close()
