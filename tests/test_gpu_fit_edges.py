"""The exact solve of the fit at the edges of its division (fit.cuh): two values, the last lengths of
the reciprocal table and the first beyond it, and values at the limits of the magnitude bound.
Records and words equal the oracle's byte for byte."""
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


def _near_limit(n):
    """Values around +-2^61 and 2^62 as int64: some partitions pass the bound, others fall back."""
    g = np.random.default_rng(31)
    base = np.repeat(g.choice(np.array([1 << 60, 1 << 61, (1 << 62) - 5000, -(1 << 61)], dtype=np.int64), n // 1000 + 1), 1000)
    return (base[:n] + g.integers(-2000, 2000, size=n)).astype(np.uint64)


DATA = {"down": lambda n: W.linear_noise(n, 1 << 50, -977, 1 << 20, seed=30), "limit": _near_limit,
        "wide": lambda n: W.random_u64(n, 32, bits=61)}


@pytest.mark.parametrize("L", [2, 3, 63, 4095, 4096, 4097, 60_000])
@pytest.mark.parametrize("kind", sorted(DATA))
def test_solve_edges_match_oracle(lc, kind, L):
    v = DATA[kind](130_003)
    rec_b, words_b, _ = lc.leco_column_export(lc.leco_encode(to_dev(v), lc.fixed(L), lc.LECO_MODEL_LINEAR))
    rec, words = oracle.encode_fixed(v, L, lc.LECO_MODEL_LINEAR)
    assert rec_b == rec.tobytes() and words_b == words.tobytes()
