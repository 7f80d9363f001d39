"""A plan's reported shape is the one that its kernels use, and planning it again gives the same plan."""
import pytest

from paper_2012_06012_gb300 import build, mgt

build.build()


@pytest.mark.parametrize("cap", [512, 5120, 5632, 8192])
@pytest.mark.parametrize("shift", [1, 5, 8, 10])
@pytest.mark.parametrize("wide", [False, True])
def test_reported_capacity(cap, shift, wide):
    """The one-block sort holds 5,120 records at most, and no more than shared memory takes."""
    args = (60_000, 60_000, 30_000_000, 2**32 if wide else 60_000_000, 8, 4)
    try:
        named = mgt.Plan(*args, cfg={"bucket_shift": shift, "cluster": 1, "chunk_cap": cap, "scatter_tile": 4096})
    except mgt.MgtError:
        assert cap > 5120 and (shift == 10 or wide)  # (refused: the widest buckets and records)
        return
    got = named.config
    assert got["chunk_cap"] <= min(cap, 5120)
    again = mgt.Plan(*args, cfg=got)
    assert again.config == got and again.workspace_bytes == named.workspace_bytes


def test_capacity_of_a_cluster_is_the_named_one():
    p = mgt.Plan(100_000, 100_000, 30_000_000, 60_000_000, 8, 4, cfg={"bucket_shift": 6, "cluster": 2, "chunk_cap": 8192})
    assert p.config["chunk_cap"] == 8192


@pytest.mark.parametrize("cols,cells", [(27, 63_108), (1, 4892), (11, 25_850), (67, 160_197), (13, 31_122)])
def test_default_shapes_of_one_column_buckets_plan_again(cols, cells):
    first = mgt.Plan(70_000, cols, cells, 5 * cells, 8, 8)
    assert first.config["bucket_shift"] == 0
    again = mgt.Plan(70_000, cols, cells, 5 * cells, 8, 8, cfg=first.config)
    assert again.config == first.config and again.workspace_bytes == first.workspace_bytes
