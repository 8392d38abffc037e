"""The encoder's paths for short partitions (a lane packs each, a tile of eight lanes fits each) and for widths
above 32 bits (rows of 64-bit entries), at the lengths where one path takes over from another. Records and words
equal the oracle's."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import to_dev

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


def _column(lens, top, seed, bits=64):
    """Values whose residual width changes from partition to partition, 0 .. top bits."""
    g = W.rng(seed)
    n = int(np.sum(lens))
    amp = np.repeat((np.uint64(1) << g.integers(0, top + 1, size=len(lens)).astype(np.uint64)) - np.uint64(1), lens)
    v = (W.random_u64(n, seed + 1) & amp) + np.uint64(1 << 10)
    return v & np.uint64(0xFFFFFFFF) if bits == 32 else v


def _check(lc, lens, v, bits, model):
    starts = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    col = lc.leco_encode_with_starts(to_dev(v, bits), to_dev(starts), len(lens), model)
    rec_b, words_b, _ = lc.leco_column_export(col)
    rec, words = oracle.encode(v, starts, model)
    assert rec_b == rec.tobytes() and words_b == words.tobytes()


@pytest.mark.parametrize("bits,top", [(64, 63), (64, 20), (32, 31)])
@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("edge", [(1, 2, 3, 4), (31, 32, 33, 34), (63, 64, 65, 66), (126, 127, 128, 129, 130)])
def test_edges_of_the_lane_path(lc, edge, model, bits, top):
    """Lengths about the limits, with a long partition now and then so that windows cut some, over means below 96,
    up to 224 and above; 64 values of 33 bits and more go beyond a lane's bits."""
    g = W.rng(100 + len(edge))
    for every, count in ((0, 3000), (40, 2000), (9, 600)):
        lens = g.choice(edge, size=count)
        if every:
            lens[::every] = g.integers(900, 5000, size=len(lens[::every]))
        _check(lc, lens, _column(lens, top, 110 + every, bits), bits, model)


@pytest.mark.parametrize("bits,top", [(64, 62), (32, 31)])
@pytest.mark.parametrize("model", [0, 1])
def test_many_short_partitions(lc, model, bits, top):
    """Enough partitions for four at a time per warp: groups of short ones, groups with a long one (256, 257, 3000
    values), a last group of one to three."""
    g = W.rng(120)
    for tail in (0, 1, 2, 3):
        lens = g.integers(1, 12, size=160_000 + tail)
        at = g.integers(0, len(lens), size=300)
        lens[at] = g.choice([255, 256, 257, 3000], size=300)
        _check(lc, lens, _column(lens, top, 121 + tail, bits), bits, model)


@pytest.mark.parametrize("bits", [33, 34, 47, 62, 63, 64])
def test_wide_pieces(lc, bits):
    """Pieces of 127 .. 129, 255 .. 257 and 511 .. 513 values at every bit of a word, and windows that cut them."""
    g = W.rng(130 + bits)
    lens = np.concatenate([g.choice([127, 128, 129, 255, 256, 257, 511, 512, 513], size=150), [1, 2, 5000, 9000]])
    v = W.random_u64(int(lens.sum()), 131 + bits, bits=bits)
    for model in (0, 1):
        _check(lc, lens, v, 64, model)


def test_32_bit_values_with_wide_residuals(lc):
    """A line through 32-bit values can leave residuals of 33 bits and more."""
    v = np.where(np.arange(70_001) % 2, 0, 0xFFFFFFFF).astype(np.uint64)
    v[::7] = W.random_u64(len(v[::7]), 140, bits=32)
    for L in (40, 300, 4096):
        col = lc.leco_encode(to_dev(v, 32), lc.fixed(L), 1)
        rec_b, words_b, _ = lc.leco_column_export(col)
        rec, words = oracle.encode_fixed(v, L, 1)
        assert rec_b == rec.tobytes() and words_b == words.tobytes()


def test_short_partitions_in_a_batch(lc):
    shapes = [(50_001, 1, 0), (40_000, 4, 1), (30_011, 33, 1), (3000, 128, 0), (20_000, 129, 1), (700, 3000, 1)]
    vals = [W.random_u64(n, 150 + k, bits=5 + 11 * k) for k, (n, _, _) in enumerate(shapes)]
    cols = lc.leco_batch_encode([to_dev(v) for v in vals], [m for _, _, m in shapes], [L for _, L, _ in shapes])
    for col, v, (_, L, model) in zip(cols, vals, shapes):
        rec_b, words_b, _ = lc.leco_column_export(col)
        rec, words = oracle.encode_fixed(v, L, model)
        assert rec_b == rec.tobytes() and words_b == words.tobytes()
