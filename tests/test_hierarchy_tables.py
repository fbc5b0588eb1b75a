"""The tables of a rebuild's launches (CoarseStates, CoarseOps in
csrc/kernels.cuh) hold every multigrid level a grid of fewer than 2^31 cells
can have: 16384x8192 cells are 13 levels, of which 12 entries hold no more
than a grid of 8192x4096."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2403_17018_gb300", "csrc")


def levels(nx, ny):
    """Levels of build_hierarchy (csrc/solver.cu)."""
    n = 1
    while nx % 4 == 0 and ny % 2 == 0 and (nx // 2) * (ny // 2) >= 8:
        nx, ny, n = nx // 2, ny // 2, n + 1
    return n


def test_every_grid_fits_the_tables():
    with open(os.path.join(CSRC, "kernels.cuh")) as f:
        src = f.read()
    size = {}
    for name in ("CoarseStates", "CoarseOps"):
        body = re.search(r"struct %s \{(.*?)\n\};" % name, src, re.S).group(1)
        used = set(re.findall(r"\[(\w+)\]", body))
        assert len(used) == 1, used
        size[name] = int(re.search(r"constexpr int %s = (\d+);" % used.pop(), src).group(1))
    shapes = [(cx << k, cy << k) for cx in range(2, 34, 2) for cy in range(1, 17) for k in range(16)
              if cx * cy <= 32 and (cx << k) * (cy << k) < 2 ** 31]
    deepest = max(levels(*s) for s in shapes)
    assert deepest == 14 and levels(16384, 8192) == 13
    assert min(size.values()) >= deepest
