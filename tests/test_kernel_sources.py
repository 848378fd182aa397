"""Rules of the kernel sources that no run on one GPU can show."""
import ctypes
import glob
import os
import re
import subprocess

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


def test_edge_copies_stay_inside_the_array(tmp_path):
    # a warp tile's copy of its edge sources, for arrays at every offset to a 16-byte boundary and every cut of them: the
    # elements read lie in the array and the wanted ones land where the gathers look for them
    src = tmp_path / "edges.cpp"
    src.write_text('''
#include "sweep_edges.cuh"
#include <algorithm>
// 0, or the first tile that reads outside [0, m) or misses an element, as 1 + ((mis * 64 + m) * 64 + b0) * 64 + b1
extern "C" int check() {
    for (int mis = 0; mis < 4; ++mis)
        for (int m = 1; m < 40; ++m)
            for (int b0 = 0; b0 < m; ++b0)
                for (int b1 = b0 + 1; b1 <= m; ++b1) {
                    int col[64];
                    std::fill(col, col + 64, -1);
                    bool ok = true;
                    auto copy = [&](int at, int e) { ok = ok && e >= 0 && e < m; col[at] = e; };
                    const int lead = dag::edge_lead(4096 + 4 * (mis + b0)), n = dag::edge_granules(lead, b1 - b0);
                    ok = ok && ((b0 - lead + mis) & 3) == 0;  // the granules start on a 16-byte boundary
                    if (dag::edge_granules_inside(lead, b0, b1, m))
                        for (int i = 0; i < 4 * n; ++i) copy(i, b0 - lead + i);
                    else {
                        ok = ok && (b0 < 3 || b1 > m - 3);
                        for (int j = 0; j < b1 - b0; ++j) copy(lead + j, b0 + j);
                    }
                    for (int e = b0; e < b1; ++e) ok = ok && col[lead + e - b0] == e;
                    if (!ok || 4 * n > (b1 - b0) + 8) return 1 + ((mis * 64 + m) * 64 + b0) * 64 + b1;
                }
    return 0;
}
''')
    lib = tmp_path / "edges.so"
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-x", "c++", "-I", CSRC, str(src), "-o", str(lib)],
                   check=True)
    assert ctypes.CDLL(str(lib)).check() == 0
    # and the kernels use this arithmetic
    code = _code(os.path.join(CSRC, "sweep_warp.cuh"))
    assert "if (edge_granules_inside(lead, c.b0, c.b1, p.m)) {" in code and code.count("wcp16(") == 2
