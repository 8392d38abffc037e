"""The packer's windows and chunks (k_encode.cu) where they can go wrong: widths 1 .. 64, windows that
split a partition inside a word, partitions longer than a window and shorter than a word, coefficient
blocks at any bit, columns at the sizes where the window shrinks. Records and words equal the oracle's."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_15374_gb300 as pkg

    pkg.build()
    oracle.build()
    from paper_2306_15374_gb300 import leco

    return leco


def _check(lc, col, v, L, model):
    rec_b, words_b, _ = lc.leco_column_export(col)
    rec, words = oracle.encode_fixed(v, L, model)
    assert rec_b == rec.tobytes() and words_b == words.tobytes()


@pytest.mark.parametrize("bits", [1, 2, 3, 5, 7, 8, 13, 16, 21, 31, 32, 33, 40, 48, 63, 64])
def test_every_width(lc, bits):
    v = W.random_u64(20_011, 40 + bits, bits=bits)
    for L in (1, 7, 300, 2049, 20_011):
        for model in (0, 1):
            _check(lc, lc.leco_encode(to_dev(v), lc.fixed(L), model), v, L, model)


@pytest.mark.parametrize("bits", [1, 11, 17, 32])
def test_32_bit_columns(lc, bits):
    v = W.random_u64(30_007, 60 + bits, bits=bits)
    for L in (3, 1000, 4096):
        _check(lc, lc.leco_encode(to_dev(v, 32), lc.fixed(L), 1), v, L, 1)


@pytest.mark.parametrize("n", [1, 255, 257, 1_245_185, 2_490_369, 4_980_739])
def test_window_sizes(lc, n):
    v = W.linear_noise(n, 1 << 20, 53, 700, seed=41)
    _check(lc, lc.leco_encode(to_dev(v), lc.fixed(1000), 1), v, 1000, 1)


@pytest.mark.parametrize("L", [64, 100, 1500, 16_384])
def test_coefficient_blocks(lc, L):
    v = W.sine_mixture(50_021, a1=1e8, p1=3000.0, a2=1e6, p2=700.0, noise=3, seed=42)
    col = lc.leco_encode(to_dev(v), lc.fixed(L), 2)
    assert L == 64 or any(np.frombuffer(lc.leco_column_export(col)[0], dtype=oracle.RECORD_DTYPE)["word3"] >> np.uint64(63))
    _check(lc, col, v, L, 2)


def test_chosen_starts(lc):
    """Partitions from one value to three windows, one after another, of every width."""
    g = W.rng(43)
    lens = np.concatenate([g.integers(1, 40, size=200), g.integers(900, 3200, size=20), [5000, 1, 1, 2, 9000]])
    g.shuffle(lens)
    starts = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    n = int(starts[-1])
    amp = np.repeat(np.uint64(1) << g.integers(0, 60, size=len(lens)).astype(np.uint64), lens)
    v = W.random_u64(n, 44) % amp + np.uint64(1 << 10)
    col = lc.leco_encode_with_starts(to_dev(v), to_dev(starts), len(lens), 1)
    rec_b, words_b, _ = lc.leco_column_export(col)
    rec, words = oracle.encode(v, starts, 1)
    assert rec_b == rec.tobytes() and words_b == words.tobytes()


def test_batch_of_windows(lc):
    vals = [W.linear_noise(n, 1 << 20, 53, 1 << k, seed=k) for k, n in enumerate((1, 4095, 4097, 100_003, 30_000, 8193))]
    Ls, models = [1, 256, 1000, 4096, 64, 10_000], [0, 1, 2, 1, 2, 1]
    for col, v, L, model in zip(lc.leco_batch_encode([to_dev(v) for v in vals], models, Ls), vals, Ls, models):
        _check(lc, col, v, L, model)


@pytest.mark.parametrize("L", [1, 255, 257, 511, 513, 1000, 1023, 1025, 1500, 2047, 2049, 1_000_003, 9_961_473, 1 << 24])
def test_windows_of_whole_partitions(lc, L):
    # windows of 256 and of 1024 positions, cut to whole partitions or a part of one
    for n in (9_961_473, 20_000_003) if L == 1000 else (9_961_473,):
        v = W.linear_noise(n, 1 << 20, 3, 700, seed=43)
        _check(lc, lc.leco_encode(to_dev(v, 32), lc.fixed(L), 1), v, L, 1)
