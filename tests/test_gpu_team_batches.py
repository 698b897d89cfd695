"""The team graph search in whole batches: CTAs that answer several queries each
(an index past the L2 line, more queries than CTAs), batches whose number of
graph searches decides on the device between the two kernels, and batches of
which the exact scan takes a part.  Answers bit for bit those of the one-warp
kernel (a call with counters takes it)."""
import numpy as np
import pytest

from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")


@pytest.mark.parametrize("storage,d,R", [(jag.JAG_VEC_F32, 100, 32), (jag.JAG_VEC_BF16, 128, 64), (jag.JAG_VEC_FP8, 120, 48)])
def test_ctas_with_several_queries(storage, d, R):
    n = 200_000
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(R)
    x = rng.standard_normal((n, d)).astype(np.float32)
    graph = rng.integers(0, n, (n, R)).astype(np.int32)
    a = np.arange(n, dtype=np.int32)      # a range of w values passes w points
    idx = jag.Index(x, attr_i32=a, R=R, graph=graph, entry=7, storage=storage)
    nq = 6 * sms
    q = torch.from_numpy(x[rng.integers(0, n, nq)] + np.float32(0.5)).cuda()
    lo = rng.integers(0, n // 2, nq).astype(np.int64)
    for m, part in ((nq, 0.0), (nq, 0.2), (nq, 0.5), (5 * sms + 1, 0.25), (17 * sms // 4, 0.0), (17 * sms // 4 + 1, 0.0), (3 * sms, 0.1)):
        w = np.where(rng.random(nq) < part, 500, n // 4)      # 500 points: scanned
        f = D.filters_range_i32(lo, lo + w - 1)[:m]
        for s0 in (0, -1):
            qm = q[:m].contiguous()
            ids, dist, _ = idx.search(qm, f, None, 10, 40, s0=s0)
            rid, rd, cnt = idx.search(qm, f, None, 10, 40, s0=s0, counters=True)
            assert torch.equal(ids, rid) and torch.equal(dist, rd)
            assert int((cnt[:, 3] == 1).sum()) == (int((w[:m] == 500).sum()) if s0 else 0)
    idx.close()


def _same_as_counted(idx, w, k, beam, **kw):
    """Batches of 1, two per SM and four per SM against the same queries counted."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    q = torch.from_numpy(w.q).cuda()
    for a, b in ((0, 1), (1, 2 * sms), (2 * sms, 5 * sms)):
        args = q[a:b].contiguous(), w.filters[a:b], w.aux, k, beam
        ids, dist, _ = idx.search(*args, s0=0, **kw)
        rid, rd, _ = idx.search(*args, s0=0, counters=True, **kw)
        assert torch.equal(ids, rid) and torch.equal(dist, rd)


@pytest.mark.parametrize("storage", [jag.JAG_VEC_F32, jag.JAG_VEC_BF16, jag.JAG_VEC_FP8])
@pytest.mark.parametrize("d,R,k,beam,hash_bits", [(20, 1, 1, 17, 0), (33, 24, 10, 33, 5), (61, 33, 10, 128, 0),
                                                  (128, 64, 20, 129, 6), (100, 48, 10, 256, 0), (200, 32, 7, 96, 0),
                                                  (600, 40, 5, 64, 0)])
def test_shapes(storage, d, R, k, beam, hash_bits):
    w = D.make_mixed(n=5000, d=d, nq=800, seed=150 + d, n_centres=10)
    idx = jag.Index.from_workload(w, R=R, l_b=32, storage=storage)
    _same_as_counted(idx, w, k, beam, hash_bits=hash_bits)
    idx.close()


def test_policy():
    w = D.make_label_zipf(n=5000, d=64, nq=800, seed=161, n_labels=40, n_centres=10)
    idx = jag.Index.from_workload(w, R=32, l_b=32, storage=jag.JAG_VEC_BF16)
    ladder = (16, 32, 64)
    theta = D.mlp_init_params(len(ladder), 4)
    theta[-1] = 0.6
    pol = jag.Policy.learned(torch.from_numpy(theta).cuda(), ladder=ladder, h0=4)
    _same_as_counted(idx, w, 10, 64, policy=pol)
    idx.close()
