"""The sparse roofline's bytes are those of the layout by groups of 32 rows,
counted here group by group and row by row (CPU only)."""
import os
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def _count(precision, rp, col):
    M, nnz = len(rp) - 1, int(rp[-1])
    v = 4 if precision == "fp32" else 8
    longer = min(200, 8 + 5 * nnz // (4 * M))
    total = 0
    for stage in range(4):
        for g in range(0, M, 32):
            rows = range(g, min(g + 32, M))
            offs = [[int(c) - r for c in col[rp[r]:rp[r + 1]]] for r in rows]
            total += 16
            if len(offs) == 32 and all(o == offs[0] for o in offs) and len(offs[0]) <= longer:
                total += 32 * len(offs[0]) * v + 4 * len(offs[0])
                continue
            total += 16 + 4 + 32
            for o in offs:
                total += len(o) * 12 + 20 if len(o) > longer else len(o) * (v + 4)
        for _ in range(M):
            total += v + 8 + 8 + v                       # x, Keff, v, the next x
            total += 8 if stage in (0, 3) else 16        # acc: written, read and written twice, read
            total += 8 if stage == 3 else 0              # v
    return total


@pytest.mark.parametrize("M", [1, 31, 32, 33, 96, 200])
@pytest.mark.parametrize("pattern", ["band", "random", "one long row", "empty rows"])
def test_layout_bytes_row_by_row(M, pattern):
    import bench
    r = np.random.default_rng(M)
    cols = []
    for s in range(M):
        if pattern == "band" or (pattern == "one long row" and s != M // 2):
            c = [x for x in (s - 1, s, s + 2) if 0 <= x < M]
        elif pattern == "one long row":
            c = list(range(M))
        elif pattern == "random":
            c = sorted(r.choice(M, int(r.integers(0, min(M, 6) + 1)), replace=False))
        else:
            c = [s] if (s // 32) % 2 else []
        cols.append(c)
    rp = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    col = np.array([x for c in cols for x in c], np.int32)
    for precision in ("fp32", "fp64"):
        assert bench.csr_layout_step_bytes(precision, rp, col) == _count(precision, rp, col)
