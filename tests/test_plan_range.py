"""Which matrices the default planner takes: up to 2^26 columns (32,768 buckets of 2,048), whatever their cells and
record width, and every plan's shape can be named again."""
import numpy as np
import pytest

import oracle
import synth
from helpers import assert_same_as_oracle, gpu_transpose
from paper_2012_06012_gb300 import build, mgt

build.build()


@pytest.mark.parametrize("cols", [1, 2**24 + 1, 2**25 - 1, 2**25, 2**25 + 1, 2**25 + 2**24, 2**26 - 1, 2**26])
@pytest.mark.parametrize("cells", [1, 40_000, 300_000_000, 2**32 - 1])
@pytest.mark.parametrize("wide", [False, True])
def test_default_plans(cols, cells, wide):
    cells = min(cells, cols * 1000)
    values = 2**32 + cells if wide else min(cells, 2**32 - 1)
    with_default = mgt.Plan(1000, cols, cells, values, 8, 4)
    named = mgt.Plan(1000, cols, cells, values, 8, 4, cfg=with_default.config)
    assert named.config["chunk_cap"] == with_default.config["chunk_cap"]
    assert with_default.workspace_bytes > 0
    if with_default.config["bucket_shift"]:  # (0 names the default width)
        assert named.config == with_default.config and named.workspace_bytes == with_default.workspace_bytes


@pytest.mark.parametrize("wide", [False, True])
def test_more_columns_are_refused(wide):
    with pytest.raises(mgt.MgtError) as e:
        mgt.Plan(1000, 2**26 + 1, 1000, 2**32 if wide else 1000, 8, 4)
    assert e.value.code == mgt.MGT_EINVAL


@pytest.mark.gpu
@pytest.mark.parametrize("cols", [2**25 + 1, 2**26])
@pytest.mark.parametrize("offset_bytes", [4, 8])
def test_transposes_of_wide_matrices(cols, offset_bytes):
    """Spread cells, and a bucket of 9,000 (chunks)."""
    rng = np.random.default_rng(cols)
    col = np.concatenate([rng.integers(0, cols, 200_000), rng.integers(cols - 1500, cols, 9000)])
    C, R = len(col), 700
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rng.integers(0, R, C), minlength=R))])
    cell_ptr = np.concatenate([[0], np.cumsum(rng.integers(0, 4, C))])
    values = rng.integers(0, 256, int(cell_ptr[-1]) * 4, dtype=np.uint8)
    x = synth.from_arrays(row_ptr, rng.permutation(col).astype(np.int32), cell_ptr, values, cols, 4,
                          offset_bytes=offset_bytes)
    assert_same_as_oracle(x, gpu_transpose(x), oracle.transpose(x))
