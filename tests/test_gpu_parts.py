"""P x P counts by each of the three ways: row blocks on super-bucket boundaries (counted by the first scatter
pass, source block by source block), blocks that cut them (the pass over the output) and more blocks than that
pass takes.  Empty blocks, one-row blocks, blocks that end inside a tile, escaped run lengths, a hot column."""
import numpy as np
import pytest

import oracle
import synth
from helpers import assert_same_as_oracle, gpu_transpose

pytestmark = pytest.mark.gpu


def _matrix(n, C, part_off, seed, hot=0.2, long_runs=0, offset_bytes=8):
    rng = np.random.default_rng(seed)
    rows = np.sort((n * rng.random(C) ** 1.5).astype(np.int64))
    col = rng.integers(0, n, C)
    col[rng.random(C) < hot] = n // 2
    lens = rng.integers(0, 4, C)
    if long_runs:
        lens[rng.integers(0, C, long_runs)] = 65_535 + rng.integers(0, 2, long_runs)
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))])
    cell_ptr = np.concatenate([[0], np.cumsum(lens)])
    values = rng.integers(0, 256, int(cell_ptr[-1]) * 4, dtype=np.uint8)
    return synth.from_arrays(row_ptr, col.astype(np.int32), cell_ptr, values, n, 4, np.asarray(part_off, np.int64),
                             offset_bytes)


def _check(x, cfg=None):
    assert_same_as_oracle(x, gpu_transpose(x, cfg=cfg), oracle.transpose(x))


@pytest.mark.parametrize("n,step,cfg", [(4096, 512, {"bucket_shift": 9, "cluster": 1}),
                                        (65_536, 256, {"bucket_shift": 4, "cluster": 1, "scatter_tile": 4096}),
                                        (40_000, 1024, {"bucket_shift": 5, "cluster": 1, "scatter_tile": 1024}),
                                        (81_920, 2560, {"bucket_shift": 2, "cluster": 1})])
@pytest.mark.parametrize("C", [1, 3072, 70_001])
def test_blocks_on_super_buckets(n, step, cfg, C):
    off = list(range(0, n, step)) + [n]
    off = sorted(off + off[2:4] * 3)  # some empty blocks
    _check(_matrix(n, C, off, C, long_runs=3 if C > 1 else 0, offset_bytes=4 if C == 3072 else 8), cfg)


@pytest.mark.parametrize("P", [2, 3, 64, 700, 2048, 2500])
@pytest.mark.parametrize("C", [5, 200_000])
def test_cut_blocks(P, C):
    n = 9001
    cuts = np.sort(np.random.default_rng(P).integers(0, n + 1, P - 1))
    _check(_matrix(n, C, np.concatenate([[0], cuts, [n]]), P, long_runs=5 if C > 5 else 0))


def test_one_row_blocks():
    _check(_matrix(600, 30_000, np.arange(601), 1))


def test_one_source_block_holds_almost_all():
    _check(_matrix(50_000, 400_000, [0, 1, 2, 49_990, 49_990, 50_000], 2, hot=0.9))
