"""What the inline PTX of the walkers promises, read from their source.

A branch with .uni states that all active threads of the warp agree on it.  The
leaders of several groups of a warp run their chains together, each with its own
predicates, so a guarded branch of the chain may promise that only where a warp has
one group.  (That wrong promise gave right results with the compiler at hand, so no
run of the kernel can show it.)
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1302_2320_gb300", "csrc")


def _sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        yield os.path.basename(path), re.sub(r"//[^\n]*", "", open(path).read())


def test_uniform_branches_only_where_a_warp_has_one_chain():
    uses = 0
    for name, src in _sources():
        for line in src.splitlines():
            if "bra.uni" not in line:
                continue
            uses += 1
            # the branch is a parameter of the chain, chosen by ALONE
            assert re.match(r"\s*if constexpr \(ALONE\) WL_CHAIN\(WL_CHAIN_\d\(\"bra\.uni\"\)\);", line), (name, line)
    assert uses <= 3
    walk = dict(_sources())["wl_walk.cuh"]
    calls = re.findall(r"chain_steps<([^>]*)>\(", walk)
    assert calls and all(re.fullmatch(r"\d, S == 32", c) for c in calls), calls
