"""The benchmark drops its recorded DRAM traffic when a solver source changes: the list of sources it hashes holds every
file that the solver's kernels are compiled from."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2003_00082_gb300", "csrc")


def includes(name, seen):
    if name in seen or "/" in name or not os.path.exists(os.path.join(CSRC, name)):
        return seen
    seen.add(name)
    with open(os.path.join(CSRC, name)) as f:
        for inc in re.findall(r'^\s*#include\s+"([^"]+)"', f.read(), re.M):
            includes(inc, seen)
    return seen


def test_hashed_sources_cover_the_solver():
    import bench
    need = set()
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cu"):
            seen = includes(f, set())
            if "cgp_solver.cuh" in seen:        # a unit with solver kernels
                need |= seen
    assert "cgp_solver.cuh" in need and need <= set(bench.SOLVER_SOURCES), sorted(need - set(bench.SOLVER_SOURCES))
