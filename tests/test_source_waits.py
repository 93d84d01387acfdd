"""Waits of the kernels that read as text must be sound, because a missing one cannot be shown
by running it: an mbarrier is initialised by one thread and polled by its warp, so a barrier of
that warp lies between the initialisation and the first poll (PTX leaves a poll of an
uninitialised mbarrier undefined)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_07488_gb300", "csrc")


def kernels():
    """(file, name, body without comments) of every kernel that initialises an mbarrier."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^{;]*?\)\s*)?(\w+)\(", src):
            i = src.index("{", m.end())
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[j], 0)
                j += 1
            if "mbar_init(" in src[i:j]:
                out.append((os.path.basename(path), m.group(1), src[i:j]))
    return out


def test_the_star_solve_is_among_them():
    assert "k_star_solve" in [name for _, name, _ in kernels()]


@pytest.mark.parametrize("path,name,body", kernels(), ids=lambda v: v if re.fullmatch(r"\w+(\.cu)?", v) else "")
def test_a_barrier_lies_between_mbarrier_init_and_the_first_poll(path, name, body):
    first, last = body.index("mbar_wait("), body.rindex("mbar_init(")
    assert last < first
    assert re.search(r"__sync(warp|threads)\(\)", body[last:first])
