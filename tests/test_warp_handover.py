"""Hand-overs inside a warp, read from the kernel sources (no GPU).

Where some lanes of a warp wait for another block's counter or a barrier and
the whole warp then reads what it guards, the vote that tells the others
(__all_sync) orders no memory by CUDA's memory model: only a __syncwarp()
between the vote and the reads makes them come after the waiting lanes'
acquire.  So every __all_sync in the kernels has one before the next load.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_13908_gb300", "csrc")
LOAD = re.compile(r"__ldcg\(|__ldg\(|ld\.|ldd2\(|ld_\w+\(|row_part\(|col_part\(|mv_\w+\(")


def _votes():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__all_sync\(", text):
            yield os.path.basename(path), text[:m.start()].count("\n") + 1, text[m.end():]


VOTES = list(_votes())


def test_the_kernels_vote():
    assert {f for f, _, _ in VOTES} == {"chol_f64.cu", "chol_solve.cu"}


@pytest.mark.parametrize("name,line,rest", VOTES, ids=["%s:%d" % v[:2] for v in VOTES])
def test_a_vote_is_followed_by_a_warp_barrier_before_any_load(name, line, rest):
    # what follows the statement that holds the vote
    rest = rest[rest.index(";") + 1:]
    sync, load = rest.find("__syncwarp()"), LOAD.search(rest)
    assert sync >= 0
    assert load is None or sync < load.start(), rest[:load.end()]
