"""Runs so long that the lengths of one warp's piece of a sorted bucket or chunk add up to more than 2^32 values
(24 GB of values; compared on the device)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap", [512, 5120], ids=["chunks", "bucket"])
@pytest.mark.parametrize("runs", [[(0, 10**9)] * 3 + [(1, 10**9)] * 3, [(0, 70_000), (1, 4_400_000_000), (1, 65_535)]],
                         ids=["six-of-1e9", "one-of-4.4e9"])
def test_sums_above_32_bits(cap, runs):
    """900 cells in a bucket of 8 columns; the long runs among the first of its first two columns."""
    import torch
    from paper_2012_06012_gb300 import mgt
    rng = np.random.default_rng(1)
    C, N, R = 900, 40, 60
    col = rng.integers(0, 8, C)
    lens = rng.integers(0, 4, C)
    col[:30] = np.arange(30) % 2
    for k, (c, n) in enumerate(runs):  # cells 0.. of column c, in the first chunk whatever its size
        at = 2 * k + c
        assert col[at] == c
        lens[at] = n
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(np.sort(rng.integers(0, R, C)), minlength=R))])
    cell_ptr = np.concatenate([[0], np.cumsum(lens)])
    V = int(cell_ptr[-1])
    order = np.argsort(col, kind="stable")
    want = np.concatenate([[0], np.cumsum(lens[order])])
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)
    values = torch.empty(V, dtype=torch.int32, device="cuda").random_()
    x = mgt.DeviceXCSR(R, N, 8, 4, dev(row_ptr, torch.int64), dev(col, torch.int32), dev(cell_ptr, torch.int64),
                       values.view(torch.uint8), np.array([0, R], np.int64))
    plan = mgt.plan_for(x, cfg={"bucket_shift": 3, "cluster": 1, "chunk_cap": cap})
    ws, out = mgt.alloc_workspace(plan.workspace_bytes), mgt.alloc_output(x, parts=False)
    mgt.transpose(plan, x.arrays(), out, ws)
    assert mgt.read_status(ws) == 0
    assert np.array_equal(out[0].cpu().numpy(), np.concatenate([[0], np.cumsum(np.bincount(col, minlength=N))]))
    assert np.array_equal(out[2].cpu().numpy(), want)
    got = out[3].view(torch.int32)
    for q, k in enumerate(order):
        a, b = int(want[q]), int(want[q + 1])
        assert torch.equal(got[a:b], values[cell_ptr[k]:cell_ptr[k + 1]]), (q, k)
    del values, got, out, x, ws
    torch.cuda.empty_cache()
