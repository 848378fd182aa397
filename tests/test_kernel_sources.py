"""Rules of the kernel sources that no run on one GPU can show."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_01409_gb300", "csrc")


def _code(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def test_no_vote_relies_on_the_lanes_that_happen_to_be_active():
    # __activemask() does not promise that lanes which diverged have met again. It may pick the lanes that share an
    # atomic (__match_any_sync: any split of the warp gives the same sums); a vote or a shuffle over it may miss some.
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for call in re.findall(r"(\w+)\(\s*__activemask\(\)", _code(path)):
            seen += 1
            assert call == "__match_any_sync", (os.path.basename(path), call)
        assert len(re.findall(r"__activemask", _code(path))) == len(re.findall(r"__match_any_sync\(\s*__activemask\(\)",
                                                                               _code(path)))
    assert seen


def test_the_warp_frontiers_marks_cannot_wrap():
    # a lane's share of a sweep's marks is added to in count_marks only, which stops it at 2^31: with one out-degree below
    # 2^31 more it still fits 32 bits (a graph that gets there is of the largest size)
    code = _code(os.path.join(CSRC, "sweep_warp_frontier.cu"))
    assert re.search(r"unsigned marks = 0u;", code)
    assert "marks +=" not in code and len(re.findall(r"count_marks\(marks,", code)) == 3
    assert "marks = min(marks + (unsigned)degree, 1u << 31);" in code and (1 << 31) + (1 << 31) - 1 < 1 << 32
