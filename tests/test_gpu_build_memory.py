"""Device memory of a Weight-JAG build: at its peak no more than a build with as
many thresholds takes (the samples of the weights are dead before the first
batch and live in memory that the batches need anyway)."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
jag = pytest.importorskip("paper_2602_10258_gb300.jag")


def _peak(**kw):
    """Most device memory in use during a build, as seen by a second thread."""
    n, d = 40_000, 16
    rng = np.random.default_rng(1)
    x = rng.standard_normal((n, d)).astype(np.float32)
    a = rng.integers(0, 1000, n).astype(np.int32)
    least, done = [], threading.Event()

    def watch():
        low = torch.cuda.mem_get_info()[0]
        while not done.is_set():
            low = min(low, torch.cuda.mem_get_info()[0])
        least.append(low)

    free = torch.cuda.mem_get_info()[0]
    t = threading.Thread(target=watch)
    t.start()
    idx = jag.Index(x, attr_i32=a, R=32, l_b=64, **kw)
    done.set()
    t.join()
    idx.close()
    return free - least[0]


def test_weights_take_no_more_memory_than_thresholds():
    _peak(thresholds=(100, 0))      # the library's own first-use allocations
    thr = max(_peak(thresholds=(100, 10, 0)) for _ in range(3))
    wgt = max(_peak(weights=(0.0, 1.0, 10.0)) for _ in range(3))
    assert wgt <= thr + (16 << 20), (thr, wgt)
