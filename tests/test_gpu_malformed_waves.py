"""Malformed inputs of many waves of blocks: blocks that start while others of the same launch flag the input
leave as a whole, so that the call reports its status, writes nothing astray and leaves the context usable."""
import numpy as np
import pytest

import oracle
import synth
from helpers import assert_same_as_oracle, gpu_transpose

pytestmark = pytest.mark.gpu


def _matrix(n=50_000, C=2_000_000, seed=4):
    rng = np.random.default_rng(seed)
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rng.integers(0, n, C), minlength=n))])
    cell_ptr = np.concatenate([[0], np.cumsum(rng.integers(0, 4, C))])
    values = rng.integers(0, 256, int(cell_ptr[-1]) * 4, dtype=np.uint8)
    return synth.from_arrays(row_ptr, rng.integers(0, n, C).astype(np.int32), cell_ptr, values, n, 4)


@pytest.mark.parametrize("cfg", [{"bucket_shift": 6, "cluster": 1, "scatter_tile": 512},
                                 {"bucket_shift": 8, "cluster": 1, "scatter_tile": 512}], ids=["two-passes", "one-pass"])
def test_cell_ptr_decreases_in_the_first_tiles(cfg):
    """3,907 tiles of which the first few flag the input: the later ones start before and after that."""
    from paper_2012_06012_gb300 import mgt
    x = _matrix()
    bad = x.cell_ptr.copy()
    for t in (0, 1, 2, 600, 700):
        bad[t * 512 + 100] = bad[t * 512 + 101] + 3
    y = synth.from_arrays(x.row_ptr, x.col_idx, bad, x.values, x.n_cols, 4)
    assert gpu_transpose(y, cfg)[6] == mgt.MGT_EBADINPUT
    assert_same_as_oracle(x, gpu_transpose(x, cfg), oracle.transpose(x))


def test_values_call_on_inconsistent_outputs():
    """The value copy checks every run that it moves; tiles that find one outside the values flag it and the
    others go on or leave, each as a whole block."""
    import torch
    from paper_2012_06012_gb300 import mgt
    x = _matrix()
    d = mgt.to_device(x)
    plan = mgt.plan_for(d)
    ws, out = mgt.alloc_workspace(plan.workspace_bytes), mgt.alloc_output(d, parts=False)
    mgt.transpose(plan, d.arrays(), out, ws)
    assert mgt.read_status(ws) == 0
    kept = out[2].clone()
    out[2][1::3] += x.n_values  # runs past the end in every tile
    mgt.transpose_values(plan, d.arrays(), out, ws)
    assert mgt.read_status(ws) == mgt.MGT_EOVERFLOW
    out[2].copy_(kept)
    mgt.transpose(plan, d.arrays(), out, ws)
    assert mgt.read_status(ws) == 0
    assert torch.equal(out[3].cpu(), torch.from_numpy(oracle.transpose(x).values))


def _device_ms(x, runs=3):
    """Fastest of a few transposes of x on the device, and the status."""
    import torch
    from paper_2012_06012_gb300 import mgt
    d = mgt.to_device(x)
    plan = mgt.plan_for(d)
    ws, out = mgt.alloc_workspace(plan.workspace_bytes), mgt.alloc_output(d, parts=False)
    best = float("inf")
    for _ in range(runs + 1):  # (the first is a warm-up)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        mgt.transpose(plan, d.arrays(), out, ws)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1])) if _ else best
    return best, mgt.read_status(ws)


def test_rows_that_claim_all_cells_again_and_again():
    """row_ptr alternates between 0 and C: every second row claims all cells.  The call is refused in no more time
    than a valid matrix of the size takes three times over (work stays linear in rows and cells)."""
    from paper_2012_06012_gb300 import mgt
    n, C = 2_000_000, 16_000_000
    col, cell_ptr = np.arange(C, dtype=np.int32) % n, np.arange(C + 1)
    values = np.zeros(C * 4, np.uint8)
    good = np.arange(n + 1) * (C // n)
    bad = np.where(np.arange(n + 1) % 2 == 1, C, 0)
    bad[n] = C
    t_good, st = _device_ms(synth.from_arrays(good, col, cell_ptr, values, n, 4))
    assert st == 0
    t_bad, st = _device_ms(synth.from_arrays(bad, col, cell_ptr, values, n, 4))
    assert st == mgt.MGT_EBADINPUT
    assert t_bad <= 3 * t_good, f"{t_bad:.2f} ms, a valid matrix takes {t_good:.2f} ms"
