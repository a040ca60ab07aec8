"""A work counter of a plan's captured adjoint launches is handed out once: a graph keeps it, and a
second graph that replayed at the same time with the same counter would skip or repeat tiles."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_1910_13555_gb300", "csrc", "adjoint.cu")


def test_no_counter_is_handed_out_twice():
    src = open(SRC).read()
    take = re.search(r"\nstatic void side_staged\(.*?\n\}", src, re.S).group(0)
    assert "next_counter.fetch_add(1)" in take  # two threads that capture draw different ones
    assert re.search(r"if \(i < kAdjCounters\) counter = S\.counters \+ i;", take)
    assert not re.search(r"next_counter[^;]*%", src)
