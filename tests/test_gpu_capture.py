"""A transpose captured into a caller's CUDA graph (after another operation in the stream), replayed on new
input data in the same buffers; many and few row blocks (offsets as a parameter or copied)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("parts", [1, 3, 300])
def test_capture_and_replay(parts):
    import torch
    from paper_2012_06012_gb300 import mgt
    spec = synth.balanced(seed=1, n=6000, parts=parts, cells=8, vals=2, stride=16, offset_bytes=4)
    xs = [synth.generate(spec), synth.generate(synth.balanced(seed=2, n=6000, parts=parts, cells=8, vals=2, stride=16,
                                                              offset_bytes=4))]
    d = mgt.to_device(xs[0])
    plan = mgt.plan_for(d)
    ws, out = mgt.alloc_workspace(plan.workspace_bytes), mgt.alloc_output(d, parts=plan.n_parts > 1)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):  # warm-up outside the graph
        mgt.transpose(plan, d.arrays(), out, ws)
    torch.cuda.synchronize()
    staged = [torch.empty_like(a) for a in d.arrays()]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for a, s in zip(d.arrays(), staged):
            a.copy_(s)
        mgt.transpose(plan, d.arrays(), out, ws)
    for x in xs:
        for s, a in zip(staged, mgt.to_device(x).arrays()):
            s.copy_(a)
        graph.replay()
        torch.cuda.synchronize()
        assert mgt.read_status(ws) == 0
        ref = oracle.transpose(x)
        want = [ref.row_ptr, ref.col_idx, ref.cell_ptr, ref.values]
        want += [ref.part_cells.reshape(-1), ref.part_values.reshape(-1)] if plan.n_parts > 1 else []
        for got, w in zip(out, want):
            assert np.array_equal(got.cpu().numpy(), w)
