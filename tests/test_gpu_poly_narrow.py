"""The polynomial model's 32-bit moments and fixed-point ranges (fit.cuh) where they can go wrong: lengths
around one lane's and one chunk's share, values at the edge of the narrow range and beyond it, predictions
that meet integers exactly, filters over sampled tile bounds. Records and words equal the oracle's."""
import numpy as np
import pytest

import oracle
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
    oracle.build()
    from paper_2306_15374_gb300 import leco

    return leco


def _cubic(n, scale, noise, seed):
    """A cubic through each 5000 values, exact when noise is 0: its residuals sit at integers."""
    x = np.arange(n, dtype=np.int64) % 5000
    y = (x - 100) * (x - 2500) * (x - 4900) // 1000 * scale + (1 << 41)
    return (y + W.rng(seed).integers(-noise, noise + 1, size=n)).astype(np.uint64)


DATA = {
    "exact": lambda n: _cubic(n, 1, 0, 50),
    "noisy": lambda n: _cubic(n, 3, 40, 51),
    "edge": lambda n: _cubic(n, 70, 7, 52),        # ranges around 2^30
    "beyond": lambda n: _cubic(n, 5000, 9, 53),
    "sine": lambda n: W.sine_mixture(n, a1=1e7, p1=9000.0, a2=1e5, p2=1100.0, noise=5, seed=54),
    "random": lambda n: W.random_u64(n, 55, bits=60),
}


@pytest.mark.parametrize("L", [64, 65, 127, 1000, 4095, 4097, 9000, 16_384])
@pytest.mark.parametrize("kind", sorted(DATA))
def test_encode_matches_oracle(lc, kind, L):
    v = DATA[kind](60_007)
    rec_b, words_b, _ = lc.leco_column_export(lc.leco_encode(to_dev(v), lc.fixed(L), 2))
    rec, words = oracle.encode_fixed(v, L, 2)
    assert rec_b == rec.tobytes() and words_b == words.tobytes()


@pytest.mark.parametrize("kind", ["exact", "noisy", "sine"])
def test_filters_over_sampled_bounds(lc, kind):
    import torch

    v = DATA[kind](200_003)
    cuts = np.sort(v)[[10, 1000, 100_000, 100_050, 199_990]]
    for L in (300, 5000, 16_384):
        col = lc.leco_encode(to_dev(v), lc.fixed(L), 2)
        for lo, hi in zip(cuts[:-1], cuts[1:]):
            for flags in (0, 1, 2):
                res = torch.zeros(3, dtype=torch.int64, device="cuda")
                lc.leco_filter_sum(col, int(lo), int(hi), res, flags)
                r = from_dev(res)
                assert (int(r[0]), int(r[1]) | int(r[2]) << 64) == exact_sum(v, int(lo), int(hi)), (L, flags)
