"""The split's speculative sweeps (k_var.cu) where they can go wrong: columns at the edges of segments
and chunks, partitions longer than a segment, sweeps that keep or change their parity, values beyond
(-2^62, 2^62), small caps, unaligned columns; forwards and seeded. Boundaries equal the oracle's."""
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


def _parity(n):
    """Noise that cuts every second value, with rare equal steps that shift which."""
    g = W.rng(21)
    v = np.cumsum(g.integers(0, 1 << 20, size=n)) + (1 << 30)
    for p in g.integers(3, max(4, n - 3), size=n // 3000 + 1):
        if p + 2 < n:
            v[p: p + 3] = v[p] + 5 * np.arange(3)
    return v.astype(np.uint64)


def _long(n):
    """A line with bounded noise 0 .. 3 whose level jumps about every 1500 values."""
    g = W.rng(22)
    step = (g.random(n) < 1 / 1500) * g.integers(1000, 1 << 24, size=n)
    return (100 + 7 * np.arange(n) + g.integers(0, 2, size=n) + np.cumsum(step)).astype(np.uint64)


def _wide(n):
    """Values on both sides of 2^63 and near 2^64, smooth for 900 values, then rough for 900."""
    g = W.rng(23)
    i = np.arange(n, dtype=np.uint64)
    rough = ((i // np.uint64(900)) % np.uint64(2)).astype(bool)
    v = np.uint64((1 << 63) - (1 << 20)) + np.uint64(37) * i
    return np.where(rough, v + g.integers(0, 1 << 62, size=n).astype(np.uint64), v)


DATA = {"line": lambda n: (np.arange(n) * 11 + 3).astype(np.uint64), "noise1": lambda n: W.linear_noise(n, 1000, 37, 1, seed=24),
        "parity": _parity, "long": _long, "wide": _wide}


def _check(lc, v, policy, tau, bits=64, lead=0, **kw):
    import torch

    d = to_dev(np.concatenate([np.zeros(lead, np.uint64), v]), bits)[lead:]
    starts = torch.empty(len(v) + 1, dtype=torch.int64, device="cuda")
    m = lc.leco_var_partition(d, starts, policy, 1)
    assert from_dev(starts)[: m + 1].tolist() == oracle.var_partition(v, tau, 1, variant="round", **kw).tolist()


@pytest.mark.parametrize("n", [1, 2, 3, 65, 511, 513, 1024, 65_535, 65_537, 66_050, 131_072 + 700])
@pytest.mark.parametrize("kind", sorted(DATA))
def test_split_matches_oracle(lc, kind, n):
    v = DATA[kind](n)
    _check(lc, v, lc.variable(0.03), 0.03)
    _check(lc, v, lc.variable(0.03, seeded=True), 0.03, seeded=True)


@pytest.mark.parametrize("kind", sorted(DATA))
@pytest.mark.parametrize("tau", [0.0, 0.1, 1.0])
def test_split_thresholds_caps_and_alignment(lc, kind, tau):
    v = DATA[kind](70_001)
    for cap in (1, 2, 31, 700):
        _check(lc, v, lc.variable(tau, cap=cap), tau, cap=cap)
    for lead in (1, 2):
        _check(lc, v, lc.variable(tau), tau, lead=lead)


@pytest.mark.parametrize("lead", [0, 1, 3])
def test_split_of_32_bit_columns(lc, lead):
    for v in (W.timestamps_u32(70_003, seed=25), W.random_u64(66_000, 26, bits=32), DATA["long"](66_000) & np.uint64(0xFFFFFFFF)):
        _check(lc, v, lc.variable(0.03), 0.03, bits=32, lead=lead)
