"""A batch of many tiny members does the work of one matrix of as many rows and cells in as many launches."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _fastest(call):
    import torch
    ms = []
    for _ in range(6):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        call()
        e[1].record()
        torch.cuda.synchronize()
        ms.append(e[0].elapsed_time(e[1]))
    return min(ms[1:])


@pytest.mark.parametrize("members", [64, 500])
def test_time_of_tiny_members(members):
    """No more than twice that matrix's time and 50 us (the launches' own fixed cost, more blocks in each)."""
    import torch
    from paper_2012_06012_gb300 import mgt
    spec = dict(cells=8, vals=4, stride=16, offset_bytes=4)
    xs = [synth.generate(synth.balanced(seed=k % 5, n=1000, parts=1, **spec)) for k in range(members)]
    ds = [mgt.to_device(x) for x in xs]
    plans = [mgt.plan_for(d) for d in ds]
    outs = [mgt.alloc_output(d, parts=False) for d in ds]
    batch = mgt.Batch(plans, [d.arrays() for d in ds], outs, mgt.alloc_workspace(mgt.batched_workspace(plans)))
    t = _fastest(batch.launch)
    refs = [oracle.transpose(x) for x in xs[:5]]
    for k, out in enumerate(outs):
        r = refs[k % 5]
        for got, want in zip(out, (r.row_ptr, r.col_idx, r.cell_ptr, r.values)):
            assert np.array_equal(got.cpu().numpy(), want), k
    one = mgt.to_device(synth.generate(synth.balanced(seed=9, n=1000 * members, parts=1, **spec)))
    plan, out = mgt.plan_for(one), mgt.alloc_output(one, parts=False)
    ws = mgt.alloc_workspace(plan.workspace_bytes)
    t_one = _fastest(lambda: mgt.transpose(plan, one.arrays(), out, ws))
    assert t <= 2 * t_one + 0.05, f"{t * 1e3:.0f} us, one matrix of the same cells {t_one * 1e3:.0f} us"
