"""Matrices with many more rows than cells: empty rows after the last cell, before the first, in one gap and
everywhere.  Bit for bit against the oracle, and in a time that follows the row pointers' bytes."""
import numpy as np
import pytest

import oracle
import synth
from helpers import assert_same_as_oracle, gpu_transpose

pytestmark = pytest.mark.gpu


def _row_ptr(kind, R, C):
    k = np.arange(C)
    rows = {"trailing": k // 4, "leading": R - 1 - k[::-1] // 4, "gap": np.where(k < C // 2, k // 4, R - 1 - (C - 1 - k) // 4),
            "spread": k * (R // C) + R // (2 * C), "clusters": k // 100 * 100 * (R // C)}[kind]
    return np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=R))])


def _matrix(kind, R, C, N=5000, offset_bytes=8, seed=0, parts=None):
    rng = np.random.default_rng(seed)
    cell_ptr = np.concatenate([[0], np.cumsum(rng.integers(0, 4, C))])
    values = rng.integers(0, 256, int(cell_ptr[-1]) * 4, dtype=np.uint8)
    return synth.from_arrays(_row_ptr(kind, R, C), rng.integers(0, N, C).astype(np.int32), cell_ptr, values, N, 4,
                             parts, offset_bytes)


KINDS = ["trailing", "leading", "gap", "spread", "clusters"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("R,C", [(3_000_001, 1), (3_000_000, 383), (2_000_003, 3073), (1_000_000, 20_000), (70_000, 384 * 9)])
def test_same_as_oracle(kind, R, C):
    x = _matrix(kind, R, C, offset_bytes=4 if C % 2 else 8, seed=C)
    assert_same_as_oracle(x, gpu_transpose(x, with_parts=False), oracle.transpose(x), check_parts=False)


@pytest.mark.parametrize("kind", KINDS)
def test_counted_source_block_by_source_block(kind):
    """Row blocks on super-bucket boundaries: pieces start at any cell."""
    n = 1 << 20
    x = _matrix(kind, n, 9000, N=n, parts=np.arange(0, n + 1, n // 32))
    assert_same_as_oracle(x, gpu_transpose(x), oracle.transpose(x))


@pytest.mark.parametrize("kind", KINDS)
def test_time_follows_the_row_pointers(kind):
    """30M rows, 3,000 cells: the row pointers are read twice (240 MB each time).  Twelve times a device copy of
    them (read and write) and half a millisecond of launches are allowed."""
    import torch
    from paper_2012_06012_gb300 import mgt
    d = mgt.to_device(_matrix(kind, 30_000_000, 3000))
    plan = mgt.plan_for(d, with_parts=False)
    ws, out = mgt.alloc_workspace(plan.workspace_bytes), mgt.alloc_output(d, parts=False)
    spare = torch.empty_like(d.row_ptr)

    def fastest(call):
        ms = []
        for _ in range(4):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            call()
            e[1].record()
            torch.cuda.synchronize()
            ms.append(e[0].elapsed_time(e[1]))
        return min(ms[1:])

    t_copy = fastest(lambda: spare.copy_(d.row_ptr))
    t = fastest(lambda: mgt.transpose(plan, d.arrays(), out, ws))
    assert mgt.read_status(ws) == 0
    assert t <= 12 * t_copy + 0.5, f"{t:.2f} ms, a copy of the row pointers takes {t_copy:.3f} ms"
