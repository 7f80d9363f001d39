"""The scatter passes' multisplit: tiles of exactly a tile's records and one more or fewer, super-buckets
that hold (nearly) all cells, long escaped runs, many and few tiles per second-pass item, wide records
between the passes.  Bit for bit against the oracle, under forced tile shapes."""
import numpy as np
import pytest

import oracle
import synth
from helpers import assert_same_as_oracle, gpu_transpose

pytestmark = pytest.mark.gpu


def _matrix(R, N, C, hot, seed, offset_bytes=8, long_runs=0):
    rng = np.random.default_rng(seed)
    rows = np.sort(rng.integers(0, R, C))
    col = rng.integers(0, N, C)
    k = int(hot * C)
    where = rng.permutation(C)[:k]
    col[where] = np.where(rng.random(k) < 0.7, N // 3, N // 3 + rng.integers(0, 3, k))  # a hot column and neighbours
    lens = rng.integers(0, 4, C)
    if long_runs:
        lens[rng.integers(0, C, long_runs)] = 65_535 + rng.integers(0, 3, long_runs)
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=R))])
    cell_ptr = np.concatenate([[0], np.cumsum(lens)])
    values = rng.integers(0, 256, int(cell_ptr[-1]) * 4, dtype=np.uint8)
    return synth.from_arrays(row_ptr, col.astype(np.int32), cell_ptr, values, N, 4, offset_bytes=offset_bytes)


def _check(x, cfg):
    assert_same_as_oracle(x, gpu_transpose(x, cfg=cfg, with_parts=False), oracle.transpose(x), check_parts=False)


@pytest.mark.parametrize("C", [1, 255, 2047, 2049, 3071, 3072, 3073, 6144, 50_001])
@pytest.mark.parametrize("hot", [0.0, 1.0])
@pytest.mark.parametrize("tile", [512, 2048, 65_536])
def test_tile_edges(C, hot, tile):
    _check(_matrix(700, 5000, C, hot, C, 4 if C % 2 else 8), {"bucket_shift": 2, "cluster": 1, "scatter_tile": tile})


@pytest.mark.parametrize("hot", [0.1, 0.6, 0.97])
@pytest.mark.parametrize("shift", [3, 6, 10])
def test_hot_super_bucket(hot, shift):
    _check(_matrix(3000, 200_000 if shift > 3 else 30_000, 300_000, hot, shift),
           {"bucket_shift": shift, "cluster": 1, "scatter_tile": 4096})


@pytest.mark.parametrize("rows", [3, 40_000, 900_000])
def test_few_and_empty_rows(rows):
    _check(_matrix(rows, 100_003, 200_000, 0.0, rows), None)


def test_escaped_runs():
    _check(_matrix(500, 9000, 20_000, 0.5, 3, long_runs=40), {"bucket_shift": 4, "cluster": 1})


def test_wide_records_between_passes():
    _check(_matrix(2000, 20_000_000, 150_000, 0.3, 9), None)
