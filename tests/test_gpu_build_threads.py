"""Index builds and network training from several threads at once, with sizes
that make the same kernels ask for different amounts of shared memory: every
call succeeds, with the results it gives alone."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")


def test_builds_of_different_sizes_at_once():
    w = D.make_range_i32(n=3000, d=128, nq=1, seed=11, width=100)
    sizes = [dict(R=64, l_b=128), dict(R=32, l_b=64), dict(R=24, l_b=32), dict(R=48, l_b=256)]

    def build(kw):
        idx = jag.Index.from_workload(w, thresholds=(100, 0), **kw)
        g = idx.graph()
        idx.close()
        return g

    alone = [build(kw) for kw in sizes]
    with ThreadPoolExecutor(len(sizes)) as ex:
        for _ in range(12):
            for a, b in zip(alone, ex.map(build, sizes)):
                assert np.array_equal(a, b)


def test_trainings_of_different_ladders_at_once():
    rng = np.random.default_rng(5)
    m = 6000
    X = torch.from_numpy(rng.standard_normal((m, 12)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.uniform(0, 3, m).astype(np.float32)).cuda()
    y = {nl: torch.from_numpy(rng.integers(0, nl, m).astype(np.int32)).cuda() for nl in (1, 5, 11, 16)}
    theta = {nl: torch.from_numpy(D.mlp_init_params(nl, nl)).cuda() for nl in y}
    torch.cuda.synchronize()

    def train(nl):
        with torch.cuda.stream(torch.cuda.Stream()):
            tr = jag.Trainer(nl, theta[nl].clone())
            for _ in range(20):
                tr.run(X, y[nl], t, 1, 3000, 1e-3, 0.5)
            return tr.params.cpu()

    alone = [train(nl) for nl in y]
    with ThreadPoolExecutor(len(y)) as ex:
        for _ in range(8):
            for a, b in zip(alone, ex.map(train, y)):
                assert torch.equal(a, b)
