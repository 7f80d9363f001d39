"""Small transposes back to back in one stream, each reading what the one before it wrote, with no wait between
them: a matrix and its transpose in turn, new values on the structure, and writes by other kernels right before."""
import numpy as np
import pytest

import oracle
import synth
from helpers import random_small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset_bytes", [4, 8])
@pytest.mark.parametrize("n", [40, 3000])
def test_there_and_back_many_times(n, offset_bytes):
    import torch
    from paper_2012_06012_gb300 import mgt
    x = random_small(n, n, n, max_cells=12, offset_bytes=offset_bytes)
    ref = oracle.transpose(x)
    a = mgt.to_device(x)
    plan = mgt.plan_for(a)
    there, back = mgt.alloc_output(a, parts=False), mgt.alloc_output(a, parts=False)
    ws = mgt.alloc_workspace(plan.workspace_bytes)
    inp, staged = [torch.zeros_like(t) for t in a.arrays()], a.arrays()
    for _ in range(60):
        for t, s in zip(inp, staged):
            t.copy_(s)
        mgt.transpose(plan, inp, there, ws)
        mgt.transpose(plan, there[:4], back, ws)
        staged = [t.clone() for t in back[:4]]
    assert mgt.read_status(ws) == 0
    for got, want in zip(there, (ref.row_ptr, ref.col_idx, ref.cell_ptr, ref.values)):
        assert np.array_equal(got.cpu().numpy(), want)
    for got, want in zip(back, (x.row_ptr, x.col_idx, x.cell_ptr, x.values)):
        assert np.array_equal(got.cpu().numpy(), want)


def test_values_written_right_before_each_copy():
    import torch
    from paper_2012_06012_gb300 import mgt
    x = random_small(5, 2000, 2000, max_cells=12, stride=8)
    a = mgt.to_device(x)
    plan = mgt.plan_for(a)
    out, ws = mgt.alloc_output(a, parts=False), mgt.alloc_workspace(plan.workspace_bytes)
    mgt.transpose(plan, a.arrays(), out, ws)
    first = out[3].view(torch.int64).clone()
    vals = a.values.view(torch.int64)
    for k in range(1, 60):
        vals += 1
        mgt.transpose_values(plan, a.arrays(), out, ws)
        if k % 20 == 0:
            assert torch.equal(out[3].view(torch.int64), first + k)
    assert mgt.read_status(ws) == 0
