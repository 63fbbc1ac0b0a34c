"""The full Wilson operator maps its thread index over full_sites(Vh), idle threads of a ragged
last warp included: every launch of it sizes its grid by that. Checked on the source text."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1109_2935_gb300", "csrc")


def test_full_operator_grids_count_full_sites():
    found = 0
    for f in sorted(os.listdir(CSRC)):
        s = open(os.path.join(CSRC, f)).read()
        # the function around each launch of wilson_kernel<.., true>
        for m in re.finditer(r"wilson_kernel<[^>;]*\btrue>", s):
            head = s[:m.start()]
            body = head[max(head.rfind("\nvoid "), head.rfind("\nstatic ")):]
            found += 1
            assert re.search(r"\bn = [^;]*full_sites\(", body), f
    assert found >= 4
