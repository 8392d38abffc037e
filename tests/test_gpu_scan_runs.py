"""The scan's runs (k_scan.cu) where they can go wrong: widths 0 .. 64 in 32- and 64-bit columns, partitions
that begin before their tile or end inside a group, more partitions per tile than are staged, ranges that
begin and end anywhere, filters at the limits of the column's width. Values and sums equal the input's."""
import numpy as np
import pytest

import workloads as W
from gpu_util import exact_sum, from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2306_15374_gb300 as pkg

    pkg.build()
    from paper_2306_15374_gb300 import leco

    return leco


def _check(lc, col, v, bits):
    import torch

    n = len(v)
    g = W.rng(70)
    tdt = torch.int32 if bits == 32 else torch.int64
    cuts = sorted({0, n, *(int(x) for x in g.integers(0, n + 1, size=4)), min(n, 4096), min(n, 4097)})
    for a in cuts:
        for b in cuts:
            if a < b:
                out = torch.empty(b - a, dtype=tdt, device="cuda")
                lc.leco_decode_range(col, a, b - a, out)
                assert (from_dev(out) == v[a:b]).all(), (a, b)
    s = np.sort(v)
    full = (1 << bits) - 1
    for lo, hi in ((0, full), (int(s[0]), int(s[0])), (int(s[n // 3]), int(s[2 * n // 3])), (int(s[-1]), (1 << 64) - 1),
                   (full, full), (1 << 33, 1 << 40), (5, 4)):
        for flags in (0, 1, 2):
            res = torch.zeros(3, dtype=torch.int64, device="cuda")
            lc.leco_filter_sum(col, lo, hi, res, flags)
            r = from_dev(res)
            assert (int(r[0]), int(r[1]) | int(r[2]) << 64) == exact_sum(v, lo, hi), (lo, hi, flags)
    assert lc.leco_sync(col) == lc.LECO_OK


@pytest.mark.parametrize("bits,width", [(64, w) for w in (0, 1, 2, 7, 31, 32, 33, 50, 63, 64)] + [(32, w) for w in (0, 1, 15, 31, 32)])
def test_widths(lc, bits, width):
    v = W.random_u64(20_011, 80 + width, bits=width) if width else np.full(20_011, 77, np.uint64)
    for L in (37, 64, 1000, 4096, 9000):
        for model in (0, 1):
            _check(lc, lc.leco_encode(to_dev(v, bits), lc.fixed(L), model), v, bits)


@pytest.mark.parametrize("bits", [32, 64])
def test_mixed_partitions(lc, bits):
    """Partitions of 1 to 9000 values, constant, smooth and noisy in turn."""
    g = W.rng(71)
    lens = np.concatenate([g.integers(1, 60, size=300), g.integers(100, 5000, size=12), [9000, 1, 31, 32, 33]])
    g.shuffle(lens)
    starts = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    n = int(starts[-1])
    amp = np.repeat(np.uint64(1) << g.choice(np.array([0, 1, 8, 17, 24]), size=len(lens)).astype(np.uint64), lens)
    v = (W.random_u64(n, 72) % amp + np.arange(n, dtype=np.uint64) * np.uint64(3)) & np.uint64((1 << bits) - 1)
    for model in (1, 2):
        _check(lc, lc.leco_encode_with_starts(to_dev(v, bits), to_dev(starts), len(lens), model), v, bits)
