"""Scratch of SCAN_ALL: bounded for few points and many queries, no larger for a
smaller batch (so that a captured call finds what a larger one left), and never
allocated while the stream is captured."""
import numpy as np
import pytest

from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")

ALL = jag.JAG_SEARCH_SCAN_ALL


def _index(n, d, seed, **kw):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((n, d)).astype(np.float32)
    return jag.Index(x, attr_f32=rng.random(n, dtype=np.float32), R=1, graph=np.full((n, 1), -1, np.int32), **kw)


def _batch(nq, d, seed):
    rng = np.random.default_rng(seed)
    q = torch.from_numpy(rng.standard_normal((nq, d)).astype(np.float32)).cuda()
    lo = (0.5 * rng.random(nq)).astype(np.float32)
    return q, jag.filters_to_device(D.filters_range_f32(lo, lo + np.float32(0.3)), "cuda")


def _captured(idx, q, f, k, stream):
    """The answers of a captured and replayed SCAN_ALL on the stream."""
    ids = torch.zeros((len(q), k), dtype=torch.int32, device="cuda")
    dist = torch.zeros((len(q), k), dtype=torch.float32, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        jag.jag_search(idx.h, q, f, None, k, k, ids, dist, stream=stream, flags=ALL)
    g.replay()
    torch.cuda.synchronize()
    return ids, dist


@pytest.mark.parametrize("storage", [jag.JAG_VEC_F32, jag.JAG_VEC_FP8])
def test_many_queries_on_few_points(storage):
    n, d, nq, k = 2100, 4, 255_000, 10      # two groups or three
    idx = _index(n, d, 1, storage=storage)
    q, f = _batch(nq, d, 2)
    ids = torch.empty((nq, k), dtype=torch.int32, device="cuda")
    dist = torch.empty((nq, k), dtype=torch.float32, device="cuda")
    idx.search(q[:10].contiguous(), f[:160].contiguous(), None, k, k, flags=ALL)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    jag.jag_search(idx.h, q, f, None, k, k, ids, dist, flags=ALL)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 1_100_000_000 + 32 * nq + n // 2 + (4 << 20)
    some = slice(nq - 300, nq)
    ri, rd, _ = idx.search(q[some].contiguous(), f.view(-1, 16)[some].contiguous(), None, k, k, flags=ALL)
    assert torch.equal(ids[some], ri) and torch.equal(dist[some], rd)
    idx.close()


def test_capture_after_a_larger_batch():
    n, d, k = 600_000, 4, 10
    idx = _index(n, d, 3)
    q, f = _batch(500, d, 4)        # two groups; a batch of 400 is one
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        want = idx.search(q, f, None, k, k, flags=ALL)
    torch.cuda.synchronize()
    ids, dist = _captured(idx, q[:400].contiguous(), f[:6400].contiguous(), k, stream)
    assert torch.equal(ids, want[0][:400]) and torch.equal(dist, want[1][:400])
    idx.close()


def test_capture_with_the_scratch_of_a_plain_search():
    n, d, k = 600_000, 4, 10
    idx = _index(n, d, 5)
    q, f = _batch(200, d, 6)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        idx.search(q, f, None, k, k)      # enough for the scan without tensor cores
        ids = torch.empty((100, k), dtype=torch.int32, device="cuda")
        dist = torch.empty((100, k), dtype=torch.float32, device="cuda")
        jag.jag_search_noalloc(idx.h, q[:100].contiguous(), f[:1600].contiguous(), None, k, k, ids, dist, flags=ALL)
    torch.cuda.synchronize()
    got = _captured(idx, q[:100].contiguous(), f[:1600].contiguous(), k, stream)
    assert torch.equal(got[0], ids) and torch.equal(got[1], dist)
    idx.close()


def test_capture_of_both_kernels():
    """Boolean filters past their line go to the brute-force kernel on a second
    stream, beside the others' scan: forked and joined inside the capture."""
    n, d, k, nq = 9000, 16, 10, 400
    rng = np.random.default_rng(7)
    idx = _index(n, d, 7, attr_mask=rng.integers(0, 1 << 12, n).astype(np.uint64))
    f, aux = D.random_bool_filters(rng, nq, 12, 4)
    lo = (0.5 * rng.random(nq)).astype(np.float32)
    f[::2] = D.filters_range_f32(lo, lo + np.float32(0.3))[::2]
    ft, at = jag.filters_to_device(f, "cuda"), jag.aux_to_device(aux, "cuda")
    q = torch.from_numpy(rng.standard_normal((nq, d)).astype(np.float32)).cuda()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        want = idx.search(q, ft, at, k, k, flags=ALL)
    torch.cuda.synchronize()
    ids, dist = torch.zeros_like(want[0]), torch.zeros_like(want[1])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        jag.jag_search(idx.h, q, ft, at, k, k, ids, dist, stream=stream, flags=ALL)
    for _ in range(2):
        ids.zero_()
        dist.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(ids, want[0]) and torch.equal(dist, want[1])
    idx.close()
