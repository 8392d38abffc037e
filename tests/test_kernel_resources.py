"""Registers of kernels whose speed is the number of warps in flight, as the compiler reports them
(no GPU needed)."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def resources(tmp_path_factory):
    from paper_2306_15374_gb300 import builder

    def go(source):
        obj = str(tmp_path_factory.mktemp("obj") / "t.o")
        cmd = [builder.nvcc(), *builder.NVCC_FLAGS, "-Xptxas", "-v", "-c", os.path.join(builder.CSRC, source), "-o", obj]
        text = subprocess.run(cmd, check=True, capture_output=True, text=True).stderr
        out = {}
        for part in text.split("Compiling entry function ")[1:]:
            out[part.split("'")[1]] = dict(regs=int(re.search(r"Used (\d+) registers", part)[1]),
                                           spills=sum(int(x) for x in re.findall(r"(\d+) bytes spill", part)))
        return out

    return go


def test_lookups(resources):
    """65536 registers hold three CTAs of 256 threads up to 80 registers a thread, four up to 64: a lookup
    waits on its loads, and a fixed column never runs the search that a variable one needs."""
    got = {k: v for k, v in resources("k_decode.cu").items() if "k_random_access" in k}
    assert len(got) == 4 and all(v["spills"] == 0 for v in got.values())
    regs = sorted(v["regs"] for v in got.values())
    assert regs[1] <= 64 and regs[3] <= 80, got  # variable partitions (two lookups per thread), fixed ones (four)
