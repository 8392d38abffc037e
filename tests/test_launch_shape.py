"""Host-side launch shapes (csrc/launch_shape.cuh), compiled by themselves: no GPU needed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2306_15374_gb300", "csrc")


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")

    def go(name, body):
        d = tmp_path_factory.mktemp(name)
        src, exe = str(d / "t.cpp"), str(d / "t")
        with open(src, "w") as f:
            f.write('#include <stdio.h>\n#include <thread>\n#include <vector>\n#include "launch_shape.cuh"\n'
                    "using namespace leco;\nint main() {\n" + body + "\nreturn 0;\n}\n")
        subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-Wall", "-Werror", "-I", CSRC, src, "-o", exe], check=True)
        return [int(x) for x in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()]

    return go


def test_every_size_is_asked_once(run):
    """Columns of every width in turn (stages of 512 bytes a bit), two devices: one question per size and
    device however often the sizes alternate."""
    asks, wrong = run("cache", """
  static ResidentCache cache;
  int asks = 0, wrong = 0;
  for (int round = 0; round < 50; round++)
    for (uint32_t b = 0; b <= 64; b++)
      for (int dev = 0; dev < 2; dev++) {
        const uint32_t smem = 1536 + 2 * (512 * b + 64 + 2048);
        const int want = 1 + (int)((b + dev) % 7);
        wrong += cache.get(dev, smem, [&]() { asks++; return want; }) != want;
      }
  printf("%d %d", asks, wrong);""")
    assert asks == 2 * 65 and wrong == 0


def test_answers_are_the_size_asked_for(run):
    """Sizes that share a slot, devices beyond the table, failures and threads: always the answer for the size."""
    wrong, asks, failed = run("mixed", """
  static ResidentCache cache;
  int wrong = 0, asks = 0;
  for (int round = 0; round < 3; round++)
    for (uint32_t smem : {2048u, 2049u, 2048u + 256u * 1024u, 3000u}) {
      for (int dev : {0, 63, 64, -1}) wrong += cache.get(dev, smem, [&]() { return (int)(smem % 251u) + 1; }) != (int)(smem % 251u) + 1;
    }
  for (int k = 0; k < 3; k++) cache.get(5, 4096, [&]() { asks++; return k < 2 ? 0 : 3; });
  const int failed = cache.get(5, 4096, []() { return -1; });
  std::vector<std::thread> ts;
  std::vector<int> bad(4);
  for (int t = 0; t < 4; t++)
    ts.emplace_back([&bad, t]() {
      for (int k = 0; k < 20000; k++) {
        const uint32_t smem = 512u * (uint32_t)((k * 7 + t) % 400);
        bad[t] += cache.get(1, smem, [&]() { return (int)(smem >> 9) % 255 + 1; }) != (int)(smem >> 9) % 255 + 1;
      }
    });
  for (auto& t : ts) t.join();
  for (int b : bad) wrong += b;
  printf("%d %d %d", wrong, asks, failed);""")
    assert wrong == 0 and asks == 3 and failed == 3


def test_small_columns_get_windows_for_many_warps(run):
    """A few thousand values are packed by as many warps as windows of 256 positions give; a large column or batch
    keeps the long ones."""
    got = run("window", """
  for (uint64_t n : {0ull, 1ull, 3000ull, 1245183ull, 5000000ull, 20000000ull, 79691776ull, 200000000ull})
    printf("%u %u %u ", pack_window(n, 4096, 256, 152 * 128), pack_window(n, 4096, 256, 152 * 32), pack_window(n, 1024, 256, 152 * 32));""")
    assert got[0::3] == [256, 256, 256, 256, 256, 1024, 4096, 4096]
    assert got[1::3] == [256, 256, 256, 256, 1024, 4096, 4096, 4096]
    assert got[2::3] == [256, 256, 256, 256, 1024, 1024, 1024, 1024]


def test_long_partitions_are_dealt_out(run):
    """Groups of eight partitions stay together where they are short or where the longest is half a pair's
    share; otherwise as many parts as that takes, a partition at the least."""
    pairs = 152 * 3 * 4
    got = run("parts", f"""
  struct {{ uint64_t values; uint32_t longest; }} cases[] = {{{{0, 0}}, {{200000000, 512}}, {{5000, 513}}, {{5000000, 4096}},
      {{16000000, 1024}}, {{50000000, 4096}}, {{100000000, 2048}}, {{100000000, 1000}}, {{200000000, 4096}}, {{1ull << 40, 1u << 24}}}};
  for (auto c : cases) printf("%u ", fit_parts(c.values, {pairs}, c.longest, 512));""")
    assert got == [1, 1, 8, 8, 2, 4, 1, 1, 1, 1]


def test_lanes_by_mean_and_window(run):
    got = run("lanes", """
  for (uint64_t mean : {0ull, 1ull, 96ull, 97ull, 224ull, 225ull, 1ull << 24})
    printf("%u %u ", lane_part_of(mean, 4096, 13), lane_part_of(mean, 256, 0));""")
    assert got == [128, 32] * 3 + [32, 32] * 2 + [0, 0] * 2
    assert run("wide", 'printf("%u %u", lane_part_of(48, 4096, 64), lane_part_of(49, 4096, 64));') == [128, 0]


def test_tried_fit_shapes_differ(run):
    """The tuner times no two shapes that start the same launch, and an older table's 4 is its 3."""
    got = run("ctas", """
  for (int most : {3, 4})
    for (uint32_t asked : {0u, 1u, 2u, 3u, 4u, 5u}) printf("%d ", fit_ctas_of(asked, most));
  for (uint32_t c : kFitCtasTried) printf("%d ", fit_ctas_of(c, 3));""")
    assert got[:6] == [3, 3, 2, 3, 3, 3] and got[6:12] == [4, 4, 2, 4, 4, 4]
    assert len(set(got[12:])) == len(got[12:]) == 2
