"""The sources whose hash ties the committed profile to the query path's code are
all of them: the translation units that the benchmark's fp32 search runs through
and every header of the library that these include."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2602_10258_gb300", "csrc")
UNITS = ("search.cu", "search_f32.cu", "team_f32.cu", "scan_tc.cu")


def test_query_sources_are_closed_under_inclusion():
    todo, seen = list(UNITS), set()
    while todo:
        f = todo.pop()
        if f in seen or not os.path.exists(os.path.join(CSRC, f)):
            continue
        seen.add(f)
        todo += re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, f), encoding="utf-8").read())
    assert {"paper_2602_10258_gb300/csrc/" + f for f in seen} <= set(bench.QUERY_SOURCES)
    assert all(os.path.exists(os.path.join(bench.ROOT, f)) for f in bench.QUERY_SOURCES)
