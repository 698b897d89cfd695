"""The exact scan where its approximations are at their worst: rows and queries
of 960 and 1,024 elements whose TF32 operands lose almost a whole unit in the
last of the ten fraction bits, all to the same side, and distances far below
the norms.  The nearest rows are then ranked behind thousands of others by the
approximations; the answers must still be those of the kernels that use no
tensor cores."""
import numpy as np
import pytest

from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")


@pytest.mark.parametrize("d", [960, 1024])
@pytest.mark.parametrize("scale", [1.0, 64.0])
def test_answers_at_the_bound(d, scale):
    n, nq = 9000, 40
    rng = np.random.default_rng(d)
    worst = np.float32(1.0 + 2.0 ** -10 - 2.0 ** -20)     # TF32 keeps 1.0
    sign = rng.choice([-1.0, 1.0], d).astype(np.float32)
    x = np.tile(sign, (n, 1))                             # exact in TF32: no loss on the rows' side
    near = rng.permutation(n)[:300]
    x[near] = sign * worst                                # every product loses 2^-9 of itself
    for i in range(n):                                    # distances: near rows below 2, the others above
        m = rng.integers(20, 27) if x[i, 0] != sign[0] else rng.integers(36, 44)
        at = rng.integers(1, d, m)
        x[i, at] += sign[at] * np.float32(0.25)
    q = np.tile(sign * worst, (nq, 1))
    for j in range(nq):
        at = rng.integers(0, d, 4)
        q[j, at] += sign[at] * np.float32(0.25)
    x *= np.float32(scale)
    q *= np.float32(scale)
    f = D.filters_none(nq)
    f[1::2] = D.filters_range_f32(np.zeros(nq // 2, np.float32), np.full(nq // 2, 0.5, np.float32))
    idx = jag.Index(x, attr_f32=rng.random(n, dtype=np.float32), R=1, graph=np.full((n, 1), -1, np.int32))
    qt = torch.from_numpy(q).cuda()
    for k in (1, 10, 128):
        rid = torch.empty((nq, k), dtype=torch.int32, device="cuda")
        rd = torch.empty((nq, k), dtype=torch.float32, device="cuda")
        jag.jag_search_noalloc(idx.h, qt, jag.filters_to_device(f, "cuda"), None, k, k, rid, rd, flags=jag.JAG_SEARCH_SCAN_ALL)
        ids, dist, _ = idx.search(qt, f, None, k, k, flags=jag.JAG_SEARCH_SCAN_ALL)
        assert torch.equal(ids, rid) and torch.equal(dist, rd)
        routed = np.arange(1, nq, 2)     # the ranges, as routed queries
        for counters in (False, True):   # a CTA per query, and a warp
            ids, dist, _ = idx.search(qt[routed].contiguous(), f[routed], None, k, k, s0=6000, scan_cap=6000, counters=counters)
            assert torch.equal(ids, rid[routed]) and torch.equal(dist, rd[routed])
        if k == 10:
            assert set(rid[0].tolist()) <= set(near.tolist())
    idx.close()
