"""leco_batch_decode reports what its decode recorded: a bounded wait that gave up is an error of the call
(there is no plan or column whose status word a caller could ask later), on any stream and with several
threads at once, and the next call starts from a clear word."""
import threading

import pytest

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
    from paper_2306_15374_gb300 import leco

    return leco


def _columns(lc, seed):
    import torch

    vals = [W.linear_noise(n, 1 << 20, 53, 700, seed=seed + n) for n in (1, 4097, 30_011)]
    cols = lc.leco_batch_encode([to_dev(v) for v in vals], [0, 1, 1], [64, 1000, 1024])
    return vals, cols, [torch.empty(len(v), dtype=torch.int64, device="cuda") for v in vals]


@pytest.mark.parametrize("side_stream", [False, True])
def test_timeout_is_reported(lc, side_stream):
    import torch

    st = torch.cuda.Stream() if side_stream else torch.cuda.current_stream()
    vals, cols, outs = _columns(lc, 70)
    torch.cuda.synchronize()
    assert lc.leco_selftest_batch_decode_timeout(cols, outs, 1_000, stream=st) == lc.LECO_ERR_TIMEOUT
    assert all((from_dev(o) == v).all() for o, v in zip(outs, vals))  # only the extra wait gave up
    for o in outs:
        o.zero_()
    torch.cuda.synchronize()
    lc.leco_batch_decode(cols, outs, stream=st)  # raises on any error
    assert all((from_dev(o) == v).all() for o, v in zip(outs, vals))


def test_threads_do_not_see_each_others_errors(lc):
    import torch

    work = [(torch.cuda.Stream(), *_columns(lc, 80 + 10 * t)) for t in range(2)]
    torch.cuda.synchronize()
    seen = [[], []]

    def loop(t):
        st, _, cols, outs = work[t]
        for _ in range(20):
            seen[t].append(lc.leco_selftest_batch_decode_timeout(cols, outs, 200, stream=st) if t else
                           lc.leco_batch_decode(cols, outs, stream=st) or lc.LECO_OK)

    threads = [threading.Thread(target=loop, args=(t,)) for t in range(2)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert seen == [[lc.LECO_OK] * 20, [lc.LECO_ERR_TIMEOUT] * 20]
    for _, vals, _, outs in work:
        assert all((from_dev(o) == v).all() for o, v in zip(outs, vals))
