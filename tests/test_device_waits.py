"""The kernels' waits of a whole warp (a property of the source: the ordering
they must give does not show in results that happen to come out right).

A lane's accesses are ordered behind an mbarrier phase that the lane has
observed itself. Where lane 0 observes it and hands the answer out by a shuffle,
which orders no memory accesses, the other lanes' reads and overwrites are
ordered by nothing. mbar_wait_warp lets every lane wait, so no kernel may hand
out such a wait by itself."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2609_05228_gb300" / "csrc"


def _without_comments(path):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", path.read_text(), flags=re.S)


def test_every_lane_waits():
    text = _without_comments(CSRC / "ace_device.cuh")
    body = re.search(r"bool mbar_wait_warp\(.*?\n}", text, re.S).group(0)
    assert "__all_sync(0xffffffffu, mbar_wait_or_abort(" in body and "lane" not in body


def test_no_kernel_hands_out_a_wait_by_a_bare_shuffle():
    """One exception: the tile rings, whose entry is read by the waiting lane itself."""
    found = []
    for path in sorted(CSRC.glob("*.cu")):
        for m in re.finditer(r"lane == 0\)\s*(\{[^}]*\}|[^;{]*;)", _without_comments(path)):
            if "mbar_wait" in m.group(1) and "ring_full" not in m.group(1):
                found.append(f"{path.name}: {' '.join(m.group(0).split())}")
    assert not found, found
