"""The variable-width copy's tiles: many tiles in the chained scan, tiles with very long runs (bytes or values
past the tile maps, one warp or the whole block per run), unit widths 1 to 32 bytes, zero widths and empty runs
inside one tile.  Bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _check(lens, widths, seed, N=83, offset_bytes=8):
    import torch
    from paper_2012_06012_gb300 import mgt
    rng = np.random.default_rng(seed)
    lens = np.asarray(lens)
    C, V = len(lens), int(lens.sum())
    rows = np.sort(rng.integers(0, 71, C))
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=71))])
    col = rng.integers(0, N, C).astype(np.int32)
    val_off = np.concatenate([[0], np.cumsum(rng.choice(widths, V))]).astype(np.int64)
    values = rng.integers(0, 256, int(val_off[-1]), dtype=np.uint8)
    x = synth.var_from_arrays(row_ptr, col, np.concatenate([[0], np.cumsum(lens)]), val_off, values, N,
                              offset_bytes=offset_bytes)
    d = mgt.to_device_var(x)
    plan = mgt.plan_for_var(d)
    out, out_off = mgt.alloc_output_var(d, parts=False)
    ws = mgt.alloc_workspace(plan.workspace_bytes)
    mgt.transpose_var(plan, d.arrays(), d.val_off, out, out_off, ws)
    assert mgt.read_status(ws) == 0
    ref = oracle.transpose_var(x)
    torch.cuda.synchronize()
    for got, want in zip((*out[:4], out_off), (ref.row_ptr, ref.col_idx, ref.cell_ptr, ref.values, ref.val_off)):
        assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("widths", [(1, 3), (0, 2, 5), (4, 12), (8, 24), (16, 48), (32, 64), (0,)])
@pytest.mark.parametrize("cells", [1, 63, 513, 60_000])
def test_unit_widths_and_many_tiles(widths, cells):
    _check(np.random.default_rng(cells).integers(0, 6, cells), widths, cells, offset_bytes=4 if cells == 513 else 8)


@pytest.mark.parametrize("widths,long", [((1,), 150_000), ((0, 4), 70_000), ((4, 8), 9000), ((32,), 80_000),
                                         ((0,), 100_000)])
def test_long_runs(widths, long):
    lens = np.random.default_rng(2).integers(0, 5, 3000)
    lens[[3, 1000, 2999]] = [long, long // 3, 1]
    _check(lens, widths, 5)
