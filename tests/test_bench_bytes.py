"""bench.py's model of the bytes of one V-cycle, against a count by hand on a two-level hierarchy, for a finest level in
the entry form (the first sweep reads the coarse vector, nothing is interpolated) and in the block form (it is).
"""
import os
import sys
from types import SimpleNamespace

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench  # noqa: E402

N, NC, NF, ROW, NNZ_R = 6, 2, 4, 5, 7      # every row of the finest level has ROW entries


class _Hierarchy:
    def __init__(self, block):
        self.block = block

    def levels(self):
        return 2

    def info(self, level):
        return SimpleNamespace(n=N if level == 0 else NC, coarsest=int(level == 1), nnz_r=NNZ_R,
                               block_size=self.block if level == 0 else 0)

    def export(self, level, what):
        return {"A.row_ptr": np.arange(N + 1) * ROW, "cf": np.array([1, 0, 0, 1, 0, 0], dtype=np.int8)}[what]


@pytest.mark.parametrize("w", [4, 8])
@pytest.mark.parametrize("block", [0, 2])
def test_vcycle_bytes(block, w):
    x = w                                                          # vector elements

    def matrix(rows):
        if block == 0:
            return rows * ROW * (w + 4)
        return rows * (ROW - 1) * w + rows * (ROW - 1) // block * 4 + rows * x    # values, block columns, diagonal

    convert = N * (2 * 8 + 2 * 4) if w == 4 else N * 4 * 8
    restrict = NNZ_R * (w + 4) + 8 * NC + x * N + x * NC
    coarsest = x * NC * NC + 2 * x * NC

    def sweep(rows, index, read):
        return matrix(rows) + index * N + 2 * x * rows + read * x + N * x          # b and 1 / a_ii; old, new vector

    if block:
        up = 4 * N + x * NC + x * N + sweep(NF, 4, N)
    else:
        up = sweep(NF, 8, NC)
    up += sweep(NC, 4, N) + sweep(NF, 4, N)
    assert bench.vcycle_bytes(_Hierarchy(block), w) == convert + restrict + coarsest + up
