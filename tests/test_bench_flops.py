"""bench.executed_tensor_flops counts what the contractions issue: 128 rows a tile,
columns and depth up to the next multiple of 16."""
import numpy as np
import pytest

import bench


class _Plan:
    def __init__(self, points, fns, rank=0):
        self.s = dict(sb_points=np.array([points], np.int32), sb_fns=np.array([fns], np.int32),
                      sb_rank=np.array([rank], np.int32))

    def schedule(self, which):
        return self.s


@pytest.mark.parametrize("points,fns,rank,columns", [
    (64, 128, 0, 128 * 64 + 128 * 128),                           # whole tiles
    (70, 130, 0, (128 + 128 + 16) * 80 + 128 * 144 + 16 * 16),    # H: tiles 00, 01, 11; density: blocks 0, 1
    (129, 7, 0, 16 * 144 + 2 * 16 * 16),                          # one short block, two point tiles
    (70, 130, -1, 0),                                             # a super-batch without tiles
])
def test_issued_columns_and_depth(points, fns, rank, columns):
    assert bench.executed_tensor_flops(_Plan(points, fns, rank), 8) == 8 * 2.0 * 128 * columns
