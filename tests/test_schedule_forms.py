"""Forms of the search and the small LP (csrc/vrm_schedule.cuh): the default
values leave them to the capacity, any other value of the caller's holds at
every capacity.  And the autotuner's side of it: n = 2 has no LP launch to
try, and files from before the small clouds' own forms lose the launch options
that were timed against other kernels."""
import json
import os
import shutil
import subprocess

import pytest

from paper_1508_06379_gb300 import autotune

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "vrm_schedule.cuh"
int main() {
  int block, per_sm, search, cap, load;
  while (std::scanf("%d %d %d %d %d", &block, &per_sm, &search, &cap, &load) == 5)
    std::printf("%d %d\n", (int)vrm::small_lp_form(block, per_sm, cap, load), (int)vrm::search_by_warps(search, cap, load));
}
"""
PAIRS, THREADS, WS, WIDE = range(4)
# lp_block, lp_blocks_per_sm, search_block, capacity, load -> LP form, search by warps
CASES = [
    ((128, 16, 256, 1, 0), (PAIRS, 1)),
    ((128, 16, 256, 65536, 0), (PAIRS, 1)),
    ((128, 16, 256, 65537, 0), (THREADS, 0)),
    ((128, 16, 256, 1179647, 0), (THREADS, 0)),
    ((128, 16, 256, 1179648, 0), (WIDE, 0)),
    ((128, 16, 256, 1179648, 5000000), (THREADS, 0)),
    ((128, 16, 256, 1000, 65536), (PAIRS, 1)),
    ((128, 16, 256, 1000, 65537), (THREADS, 0)),
    ((128, 8, 256, 1000, 0), (THREADS, 1)),
    ((64, 16, 256, 1000, 0), (THREADS, 1)),
    ((128, 17, 256, 2000000, 0), (THREADS, 0)),
    ((192, 2, 256, 1000, 0), (WS, 1)),
    ((384, 1, 64, 1000, 0), (WIDE, 0)),
    ((384, 16, 256, 2000000, 5000000), (WIDE, 0)),
    ((128, 16, 128, 1000, 0), (PAIRS, 0)),
]


def test_forms(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "forms.cpp", tmp_path / "forms"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_1508_06379_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    r = subprocess.run([str(exe)], input="".join("%d %d %d %d %d\n" % c for c, _ in CASES), capture_output=True,
                       text=True, check=True)
    got = [tuple(map(int, line.split())) for line in r.stdout.splitlines()]
    assert got == [want for _, want in CASES]


class FakeContext:
    """A context whose step does nothing on host tensors."""
    k_cap = 32

    def __init__(self, order):
        self.order, self.set = order, []

    def set_schedule(self, s):
        self.set.append(dict(s))

    def set_timing(self, on):
        pass

    def step(self, x, y, n, gi, go, dt, stats=True):
        return n, dict(max_count=12)

    def stage_times(self):
        return dict(search=1.0, lp_small=1.0, apply=1.0)


@pytest.mark.parametrize("order", [1, 2])
def test_the_lp_launch_is_tuned_for_order_1_only(order):
    torch = pytest.importorskip("torch")
    z = torch.zeros(4, dtype=torch.float64)
    ctx = FakeContext(order)
    best, _ = autotune.tune_context(ctx, z, z, 4, z, z, 1e-3, reps=1)
    tried = {(s["lp_block"], s["lp_blocks_per_sm"]) for s in ctx.set}
    assert (len(tried) > 1) == (order == 1)
    assert {s["lp_fp64_pivots"] for s in ctx.set} == {0, 1}
    if order == 2:
        assert (best["lp_block"], best["lp_blocks_per_sm"]) == (128, 16)


def test_old_files_lose_the_small_buckets_launch_options(tmp_path):
    path = str(tmp_path / "s.json")
    old = dict(row_cap=16, search_block=64, lp_block=32, lp_blocks_per_sm=4, apply_block=128, lp_fp64_pivots=1)
    keys = [autotune.cache_key("d", 32, 2.0 ** b) for b in (10, 16, 17)]
    json.dump({k: old for k in keys}, open(path, "w"))
    t = autotune.Autotuner(path)
    reset = dict(old, search_block=256, lp_block=128, lp_blocks_per_sm=16)
    assert [t.table[k] for k in keys] == [reset, reset, old]
    # files of today keep what was tuned
    t.table[keys[0]] = dict(old)
    t.save()
    assert autotune.Autotuner(path).table[keys[0]] == old
