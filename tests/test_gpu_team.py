"""The graph search with several warps per query against the one with a single
warp per query (a batch past eight queries per SM takes it): same answers and
hops, bit for bit, at the edges of the team kernel's ranges; and against the
oracle on a graph whose out-lists repeat vertices."""
import numpy as np
import pytest

from oracle import jag_oracle as O
from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")


def _both(idx, w, k, beam, **kw):
    """(whole batch, the same queries in batches of 1, 2 per SM and the rest)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nq = 8 * sms + 30
    q = torch.from_numpy(w.q[:nq]).cuda()
    f = w.filters[:nq]
    whole = idx.search(q, f, w.aux, k, beam, counters=True, s0=0, **kw)
    cuts = [0, 1, 1 + 2 * sms, 2 + 4 * sms, nq - 3, nq]
    parts = [idx.search(q[a:b].contiguous(), f[a:b], w.aux, k, beam, counters=True, s0=0, **kw)
             for a, b in zip(cuts, cuts[1:])]
    return whole, [torch.cat([p[i] for p in parts]) for i in range(3)]


@pytest.mark.parametrize("storage", [jag.JAG_VEC_F32, jag.JAG_VEC_BF16, jag.JAG_VEC_FP8])
@pytest.mark.parametrize("d,R,k,beam,hash_bits", [(20, 1, 1, 1, 0), (33, 24, 10, 33, 5), (61, 33, 10, 128, 0),
                                                  (128, 64, 20, 129, 6), (100, 48, 10, 256, 0), (200, 32, 7, 96, 0),
                                                  (600, 40, 5, 64, 0)])
def test_team_matches_single_warp(storage, d, R, k, beam, hash_bits):
    w = D.make_mixed(n=5000, d=d, nq=1400, seed=50 + d, n_centres=10)
    idx = jag.Index.from_workload(w, R=R, l_b=32, storage=storage)
    whole, parts = _both(idx, w, k, beam, hash_bits=hash_bits)
    assert torch.equal(whole[0], parts[0]) and torch.equal(whole[1], parts[1])
    assert torch.equal(whole[2][:, 0], parts[2][:, 0])   # hops
    idx.close()


def test_team_policy_matches_single_warp():
    w = D.make_label_zipf(n=5000, d=64, nq=1400, seed=61, n_labels=40, n_centres=10)
    idx = jag.Index.from_workload(w, R=32, l_b=32, storage=jag.JAG_VEC_BF16)
    ladder = (16, 32, 64)
    theta = D.mlp_init_params(len(ladder), 4)
    theta[-1] = 0.6
    pol = jag.Policy.learned(torch.from_numpy(theta).cuda(), ladder=ladder, h0=4)
    whole, parts = _both(idx, w, 10, 64, policy=pol)
    assert torch.equal(whole[0], parts[0]) and torch.equal(whole[1], parts[1])
    assert torch.equal(whole[2][:, 0], parts[2][:, 0])
    idx.close()


@pytest.mark.parametrize("R", [32, 64])
def test_team_repeated_edges(R):
    w = D.make_range_i32(n=2000, d=24, nq=50, seed=7, width=300)
    rng = np.random.default_rng(R)
    g = rng.integers(0, 2000, (2000, R)).astype(np.int32)
    g[:, R // 2:] = g[:, rng.integers(0, R // 2, R - R // 2)]   # half of each out-list repeats the other half
    ox = O.Index.from_workload(w, R=R, graph=g, entry=3)
    rid, rd, _ = O.query(ox, w.q, w.filters, w.aux, 10, 80, s0=0)
    idx = jag.Index.from_workload(w, R=R, graph=g, entry=3)
    for hb in (0, 5):
        ids, dist, _ = idx.search(torch.from_numpy(w.q).cuda(), w.filters, w.aux, 10, 80, s0=0, hash_bits=hb)
        assert np.array_equal(ids.cpu().numpy(), rid) and np.array_equal(dist.cpu().numpy(), rd)
    idx.close()
