"""Builds whose points unite more visited vertices than a warp's slice of shared
memory holds (eight Weight-JAG comparators that look in different places):
past the 256-candidate slice (a spill inside the first prune launch) and past
1,024 (the second launch); graphs identical to the oracle's."""
import numpy as np
import pytest

from oracle import jag_oracle as O
from paper_2602_10258_gb300 import datagen as D

pytestmark = pytest.mark.gpu

jag = pytest.importorskip("paper_2602_10258_gb300.jag")

MULT = (0.0, 0.3, 1.0, 3.0, 10.0, 100.0, 1e4, 1e6)


@pytest.mark.parametrize("n,lb", [(4000, 25), (3500, 256)])
def test_large_unions_match_the_oracle(n, lb):
    w = D.make_range_i32(n=n, d=12, nq=1, seed=70 + lb, width=100)
    ox = O.Index.from_workload(w, R=32)
    O.build_weighted(ox, mult=MULT, lb=lb)
    gi = jag.Index.from_workload(w, R=32, l_b=lb, weights=MULT)
    assert np.array_equal(gi.graph(), ox.graph)
    gi.close()
