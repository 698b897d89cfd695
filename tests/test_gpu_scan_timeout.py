"""The exact scan when its contraction gives up waiting for the tensor cores
(the wait is set to no polls at all): the approximations in the scratch are
then those of an earlier call, and the answers must not depend on them.  The
earlier queries are the mirror images of the later ones, so that they are as
far from most rows (the check of the candidates' approximations holds) and far
from the nearest ones (whose approximations would hide them).
SCAN_ALL and routed batches on both sides of the selection kernels' line,
against the scan kernels that use no tensor cores."""
import ctypes as C

import numpy as np
import pytest

from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")


def _noalloc(idx, q, f, k, **kw):
    ids = torch.empty((len(q), k), dtype=torch.int32, device="cuda")
    dist = torch.empty((len(q), k), dtype=torch.float32, device="cuda")
    jag.jag_search_noalloc(idx.h, q, jag.filters_to_device(f, "cuda"), None, k, k, ids, dist, **kw)
    return ids, dist


@pytest.mark.parametrize("nq", [40, 1500])
@pytest.mark.parametrize("scan_all", [True, False])
def test_answers_without_the_contraction(nq, scan_all):
    n, d, k = 9000, 40, 10
    rng = np.random.default_rng(nq)
    x = rng.standard_normal((n, d)).astype(np.float32)
    a = rng.random(n, dtype=np.float32)
    x[:, 0] = 0.0
    x[:20, 0], a[:20] = 10.0, 0.5
    lo = (0.32 + 0.16 * rng.random(nq)).astype(np.float32)
    f = D.filters_range_f32(lo, lo + np.float32(0.2))     # about 1,800 rows each
    q = torch.from_numpy(rng.standard_normal((nq, d)).astype(np.float32)).cuda()
    q[:, 0] = 10.0
    mirror = q.clone()
    mirror[:, 0] = -10.0
    idx = jag.Index(x, attr_f32=a, R=4, graph=np.full((n, 4), -1, np.int32))
    kw = dict(flags=jag.JAG_SEARCH_SCAN_ALL) if scan_all else dict(s0=6000, scan_cap=6000)
    idx.search(mirror, f, None, k, k, **kw)
    wait = jag.load().jag_internal_scan_wait
    wait.argtypes, wait.restype = [C.c_void_p, C.c_uint32], None
    wait(idx.h, 0)
    ids, dist, _ = idx.search(q, f, None, k, k, **kw)
    hid, hdist, _ = idx.search_host(q.cpu().numpy(), f, None, k, k, **kw)
    step = 200   # what fits the fixed scratch
    for i in range(0, nq, step):
        rid, rd = _noalloc(idx, q[i:i + step].contiguous(), f[i:i + step], k, **kw)
        assert torch.equal(ids[i:i + step], rid) and torch.equal(dist[i:i + step], rd)
        assert np.array_equal(hid[i:i + step], rid.cpu().numpy()) and np.array_equal(hdist[i:i + step], rd.cpu().numpy())
    idx.close()
