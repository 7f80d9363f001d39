"""The value copy's tiles: every unit width (32, 16, 8 and 4 bytes, by stride, run lengths and buffer
alignment), tiles with empty runs, tiles of one more and one fewer cell than a tile, tiles too long for
the unit map (one warp per run, the whole block per very long run).  Bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _matrix(n_cells, lens, stride, offset_bytes=8, seed=0):
    rng = np.random.default_rng(seed)
    R = N = 97
    rows = np.sort(rng.integers(0, R, n_cells))
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=R))])
    col = rng.integers(0, N, n_cells).astype(np.int32)
    cell_ptr = np.concatenate([[0], np.cumsum(lens)])
    values = rng.integers(0, 256, int(cell_ptr[-1]) * stride, dtype=np.uint8)
    return synth.from_arrays(row_ptr, col, cell_ptr, values, N, stride, offset_bytes=offset_bytes)


def _check(x, unroll=0, shift_in=0, shift_out=0):
    import torch
    from paper_2012_06012_gb300 import mgt
    d = mgt.to_device(x)
    nb = d.values.numel()
    big_in, big_out = (torch.zeros(nb + 64, dtype=torch.uint8, device="cuda") for _ in range(2))
    big_in[shift_in:shift_in + nb] = d.values
    out = list(mgt.alloc_output(d, parts=False))
    out[3] = big_out[shift_out:shift_out + nb]
    plan = mgt.plan_for(d, cfg={"copy_unroll": unroll} if unroll else None)
    ws = mgt.alloc_workspace(plan.workspace_bytes)
    mgt.transpose(plan, (*d.arrays()[:3], big_in[shift_in:shift_in + nb]), out, ws)
    assert mgt.read_status(ws) == 0
    ref = oracle.transpose(x)
    for got, want in zip(out[:4], (ref.row_ptr, ref.col_idx, ref.cell_ptr, ref.values)):
        assert np.array_equal(got.cpu().numpy(), want)
    guard = torch.cat([big_out[:shift_out], big_out[shift_out + nb:]])
    assert int(guard.count_nonzero()) == 0


@pytest.mark.parametrize("stride", [4, 8, 12, 16, 24, 32, 64])
@pytest.mark.parametrize("cells", [1, 31, 513, 5000])
def test_unit_widths_and_tile_edges(stride, cells):
    rng = np.random.default_rng(cells)
    _check(_matrix(cells, rng.integers(0, 9, cells), stride, 4 if cells % 2 else 8, cells))


@pytest.mark.parametrize("shift_in,shift_out", [(0, 4), (4, 0), (8, 8), (16, 0), (0, 16), (32, 32)])
def test_buffer_alignment(shift_in, shift_out):
    _check(_matrix(700, np.full(700, 4), 8), shift_in=shift_in, shift_out=shift_out)


@pytest.mark.parametrize("unroll", [1, 2, 4])
@pytest.mark.parametrize("stride,long", [(4, 40_000), (8, 3000), (32, 200_000)])
def test_long_runs(unroll, stride, long):
    lens = np.random.default_rng(1).integers(0, 40, 600)
    lens[[0, 77, 300, 599]] = [long, long // 2 + 1, 0, long - 1]
    _check(_matrix(600, lens, stride), unroll)


def test_empty_tiles():
    lens = np.zeros(4000, np.int64)
    lens[[5, 3999]] = [3, 1]
    _check(_matrix(4000, lens, 16))
