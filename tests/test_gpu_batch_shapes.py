"""Batched encodes at the shapes where the fit deals groups of partitions out in parts and the packer's windows
shrink: few long partitions, groups that mix lengths, models and columns, small columns. Records and words
equal the oracle's, by the direct call and by a plan's graph."""
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


CASES = {
    "one column of long partitions": ([(70_001, 513, 1)], 64),
    "last group of one": ([(9 * 1000, 1000, 0)], 64),
    "lengths mixed inside a group": ([(3000, 4096, 1), (700, 64, 0), (1, 1, 1), (0, 8, 1), (5000, 5000, 0), (2600, 513, 1)], 64),
    "models mixed inside a group": ([(2000, 600, 1), (1500, 600, 2), (1300, 700, 0), (400, 100, 2), (900, 900, 1)], 64),
    "32-bit": ([(30_007, 1024, 0), (300, 64, 1), (4097, 2047, 1)], 32),
    "up to 1024": ([(5_000, 513, 1), (9_001, 1024, 0), (700, 64, 1), (1, 1, 0), (2500, 600, 2), (3_333, 1023, 1)], 64),
    "up to 1024, many": ([(12_000_000, 700, 1), (50_000, 1024, 0)], 32),
    "one above 1024": ([(5_000, 513, 1), (4_100, 1025, 0)], 64),
    "parts of four": ([(9_000 * 2048, 2048, 1), (10_000, 500, 0)], 32),
    "parts of two": ([(17_000 * 2048, 2048, 0), (10_000, 100, 1)], 32),
    "small": ([(3000, 64, 1)] * 4, 64),
}


@pytest.mark.parametrize("name", CASES)
def test_shapes(lc, name):
    shapes, bits = CASES[name]
    vals = [W.linear_noise(n, 1 << 20, 3, 1 << (4 + k), seed=90 + k) for k, (n, _, _) in enumerate(shapes)]
    dev = [to_dev(v, bits) for v in vals]
    models, Ls = [m for _, _, m in shapes], [L for _, L, _ in shapes]
    plan = lc.leco_batch_encode_plan_create(dev, models, Ls)
    lc.leco_batch_encode_plan_run(plan)
    for cols in (lc.leco_batch_encode(dev, models, Ls), lc.leco_batch_encode_plan_columns(plan)):
        for col, v, L, model in zip(cols, vals, Ls, models):
            rec_b, words_b, _ = lc.leco_column_export(col)
            rec, words = oracle.encode_fixed(v, L, model)
            assert rec_b == rec.tobytes() and words_b == words.tobytes()
    lc.leco_batch_encode_plan_free(plan)
