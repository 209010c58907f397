"""Byte counts the bench line's roofline uses for the kernels of the present iteration (D + 1 components; D fields of w)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("D,fp,rows,medium", [(3, 4, 144, 20), (3, 8, 288, 40), (2, 4, 104, 16), (2, 8, 208, 32)])
def test_bytes_of_the_present_kernels(D, fp, rows, medium):
    sys.path.insert(0, ROOT)
    try:
        import bench
    finally:
        sys.path.remove(ROOT)
    cb = 2 * fp  # one complex value
    own, model = bench.kernel_bytes_per_voxel(D, fp), bench.model_bytes_per_voxel(D, fp)
    # x, y and D fields of w in, x and D fields of w out, and the medium: D + 2 arrays as stored, 3 in the model
    assert own["rows_update"] == rows + medium
    assert model["rows_update"] == rows + 3 * fp
    for b in (own, model):
        assert b["axis_merge"] == b["axis_split"] == 5 * cb
        assert b["last_solve"] == 4 * cb
