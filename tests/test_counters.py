"""Every per-leg counter that a leg's totals report is counted somewhere: one
that nothing increments would make the checks on it pass whatever happens."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2004_11040_gb300", "csrc")


def test_reported_counters_are_counted():
    text = open(os.path.join(CSRC, "graph.cu")).read()
    reported = set(re.findall(r"\blc\[(LC_\w+)\]", text)) - {"LC_N"}
    counted = set(re.findall(r"atomicAdd\([\w\.\[\]]+ \+ (LC_\w+),", text))
    counted |= set(re.findall(r"lc\[(LC_\w+)\] \+=", text))
    assert len(reported) >= 10
    assert reported <= counted, reported - counted
