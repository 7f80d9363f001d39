"""The per-bucket sort: buckets of exactly a block's capacity and one more (two chunks), chunks of hot
columns, narrow to 2,048-column buckets, empty buckets, escaped run lengths inside buckets and chunks,
capacities above what the one-block sort takes.  Bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from helpers import assert_same_as_oracle, gpu_transpose

pytestmark = pytest.mark.gpu


def _check(cols, N, cfg, lens=None, offset_bytes=8, stride=4, seed=0):
    """cols: the cells' columns in input order, dealt to ascending rows."""
    rng = np.random.default_rng(seed)
    C, R = len(cols), 301
    rows = np.sort(rng.integers(0, R, C))
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=R))])
    lens = rng.integers(0, 5, C) if lens is None else lens
    cell_ptr = np.concatenate([[0], np.cumsum(lens)])
    values = rng.integers(0, 256, int(cell_ptr[-1]) * stride, dtype=np.uint8)
    x = synth.from_arrays(row_ptr, np.asarray(cols, np.int32), cell_ptr, values, N, stride, offset_bytes=offset_bytes)
    assert_same_as_oracle(x, gpu_transpose(x, cfg=cfg, with_parts=False), oracle.transpose(x), check_parts=False)


def _full_buckets(n, w, buckets, seed):
    """n cells in every other bucket of w columns, in random order (the others are empty)."""
    rng = np.random.default_rng(seed)
    cols = np.concatenate([b * 2 * w + rng.integers(0, w, n) for b in range(buckets)])
    return rng.permutation(cols)


@pytest.mark.parametrize("cap", [512, 1024, 5120, 8192])
@pytest.mark.parametrize("over", [-1, 0, 1, 600])
@pytest.mark.parametrize("shift", [0, 5, 8])
def test_capacity_edges(cap, over, shift):
    w = 1 << shift
    cols = _full_buckets(cap + over, w, 7, cap + over)
    _check(cols, 14 * w, {"bucket_shift": shift or 1, "cluster": 1, "chunk_cap": cap}, offset_bytes=4 if over else 8)


@pytest.mark.parametrize("shift", [9, 10, 11])
def test_wide_buckets(shift):
    rng = np.random.default_rng(shift)
    cols = np.concatenate([rng.integers(0, 9000, 30_000), np.full(9000, 4444)])
    _check(rng.permutation(cols), 9000, {"bucket_shift": shift, "cluster": 1, "chunk_cap": 1024})


@pytest.mark.parametrize("cluster", [1, 2])
def test_escaped_lengths_in_buckets_and_chunks(cluster):
    rng = np.random.default_rng(3)
    cols = rng.permutation(np.concatenate([rng.integers(0, 64, 3000), np.full(2500, 200), rng.integers(192, 256, 500)]))
    lens = rng.integers(0, 4, len(cols))
    lens[rng.integers(0, len(cols), 12)] = 65_535
    lens[np.flatnonzero(cols == 200)[[0, 5, 2499]]] = [65_536, 70_000, 65_534]
    _check(cols, 300, {"bucket_shift": 6, "cluster": cluster, "chunk_cap": 512}, lens)


@pytest.mark.parametrize("N", [1, 13, 48])
def test_few_long_columns(N):
    _check(np.random.default_rng(N).integers(0, N, 60_000), N, None)


@pytest.mark.parametrize("N", [1025, 9000])
def test_many_chunks_and_work_list_blocks(N):
    """More than 1,024 buckets (several blocks build the work list), a bucket of over 512 chunks and some of a few."""
    rng = np.random.default_rng(N)
    cols = np.concatenate([rng.integers(0, N, 30_000), np.full(300_000, N - 1), np.full(3000, 7), np.full(1500, N // 2)])
    _check(rng.permutation(cols), N, {"bucket_shift": 1 if N > 2000 else 0, "cluster": 1, "chunk_cap": 512,
                                      "scatter_tile": 16384})
