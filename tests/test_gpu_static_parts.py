"""P x P counts through the allocation-free entry point, whose scatter pass counts them per cell in shared memory
(up to 256 row blocks): tiles of several rounds, the largest tiles (near the scratch limit), tiles that span two
and more source blocks, cut and whole super-buckets, empty blocks, escaped run lengths.  Bit for bit against the
oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _run(n, C, part_off, seed, order):
    import torch
    from paper_2012_06012_gb300 import mgt
    rng = np.random.default_rng(seed)
    rows = rng.random(C) ** order * n  # order 1: even rows; larger: most cells in the first rows
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows.astype(np.int64), minlength=n))])
    col = rng.integers(0, n, C)
    col[rng.random(C) < 0.1] = n // 2
    lens = rng.integers(0, 3, C)
    lens[rng.integers(0, C, 6)] = 65_535 + rng.integers(0, 2, 6)
    cell_ptr = np.concatenate([[0], np.cumsum(lens)])
    values = rng.integers(0, 256, int(cell_ptr[-1]) * 4, dtype=np.uint8)
    x = synth.from_arrays(row_ptr, col.astype(np.int32), cell_ptr, values, n, 4, np.asarray(part_off, np.int64), 8)
    d, ref = mgt.to_device(x), oracle.transpose(x)
    out = mgt.alloc_output(d, parts=True)
    want = (ref.row_ptr, ref.col_idx, ref.cell_ptr, ref.values, ref.part_cells.reshape(-1), ref.part_values.reshape(-1))
    for _ in range(3):
        for t in out:
            t.fill_(0x5A if t.dtype == torch.uint8 else -7)
        mgt.transpose_static(d, d.arrays(), out)
        assert mgt.static_status() == 0
        for name, a, b in zip(mgt._OUT_NAMES, out, want):
            assert np.array_equal(a.cpu().numpy(), b), name


# 2.30M cells: tiles of 6,144 cells (two rounds); 2.37M cells fit the scratch with the largest tiles alone
# (86 rounds, nine tiles); 2,000 columns: a single scatter pass
@pytest.mark.parametrize("n,C", [(300_000, 2_300_000), (300_000, 2_370_000), (2000, 2_300_000)])
@pytest.mark.parametrize("P", [2, 64, 256])
@pytest.mark.parametrize("order", [1, 6])
def test_counts_of_several_rounds_per_tile(n, C, P, order):
    cuts = np.sort(np.random.default_rng(P).integers(0, n + 1, P - 1))
    if P > 2:
        cuts[P // 2] = cuts[P // 2 - 1]  # an empty block
    _run(n, C, np.concatenate([[0], cuts, [n]]), P + C, order)


def test_counts_of_whole_super_buckets():
    n = 256 * 1024
    _run(n, 2_300_000, np.arange(0, n + 1, n // 64), 7, 2)
