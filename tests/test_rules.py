"""The launch rules (csrc/rules.h) that are plain arithmetic, built by the host compiler.

* a round of the tail's events always goes on, up to the last event number;
* the tail kernel has draw slots at every bin count, and every table that has
  room in 200 KB without them;
* so have the main kernel's warps their batches, in blocks below 1024 threads.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "rules.h"
using namespace mcbte;
int main() {
  // lines of "<rule> <arguments>" on the standard input
  char rule[32];
  unsigned a[8];
  auto take = [&](int k) { for (int i = 0; i < k; ++i) if (scanf("%u", &a[i]) != 1) exit(1); };
  auto show = [](const SmemPlan& S) {
    printf("%d %d %d %d %d %d %d %zu\n", S.relax_in_smem, S.binf_in_smem, S.cells_in_smem, S.qbin_in_smem,
           S.grad_in_smem, S.snap_in_smem, S.tail_slots + S.batch_slots, S.bytes);
  };
  while (scanf("%31s", rule) == 1) {
    if (!strcmp(rule, "round_end")) {
      take(3);
      printf("%u\n", round_end(a[0], a[1], a[2]));
    } else if (!strcmp(rule, "plan_tail")) {
      take(6);
      show(plan_tail(a[0], a[1], a[2], a[3], a[4], a[5]));
    } else if (!strcmp(rule, "plan_main")) {
      take(8);
      show(plan_main(a[0], a[1] != 0, a[2], a[3], a[4], a[5], a[6], a[7]));
    }
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, exe = d / "driver.cpp", d / "driver"
    src.write_text(DRIVER)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-I",
                           os.path.join(ROOT, "paper_2104_03573_gb300", "csrc"), "-o", str(exe), str(src)])

    def call(rule, calls):
        text = "\n".join(" ".join([rule, *map(str, c)]) for c in calls)
        out = subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout
        return [[int(x) for x in line.split()] for line in out.splitlines()]
    return call


@pytest.mark.parametrize("max_events", [1, 2, 64, 777, 2 ** 31, 2 ** 32 - 64, 2 ** 32 - 2, 2 ** 32 - 1])
@pytest.mark.parametrize("span", [1, 2, 32, 64, 65536])
def test_tail_rounds_go_on_to_the_last_event(rules, span, max_events):
    last = max_events - 1
    starts = sorted({e for e in (0, 1, last - 2 * span, last - span - 1, last - span, last - span + 1, last - 2,
                                 last - 1, last) if 0 <= e <= last})
    got = rules("round_end", [(e, span, max_events) for e in starts])
    for e, (end,) in zip(starts, got):
        assert end == min(e + span, last)
        assert end > e or e == last


KB = 1024
BINS = sorted({*range(1, 20_000, 7), *range(20_000, 70_000, 501), 3000, 5120, 5121, 6400, 6401, 12_800, 12_801, 25_600,
               65_536, 65_537})


def _tables(n, G, nc, pb, grad, snap, budget=200 * KB):
    """Tables and tallies placed one after the other while they fit, and their bytes."""
    used, res = 0, []
    for wanted, size in ((True, 16 * n), (True, 16 * n), (nc > 0 and G == 1, (8 * nc + 4) * 8), (pb and G == 1, 8 * n),
                         (grad, 8 * n), (snap > 0, 64 * snap)):
        res.append(int(bool(wanted) and used + size <= budget))
        used += size * res[-1]
    return res, used


# forward, its cells and per-bin flux, a batch of geometries, gradients
ASKS = [(1, 0, 0, 0, 0), (1, 50, 1, 0, 0), (1, 50, 0, 0, 0), (1, 1500, 1, 0, 0), (1, 4096, 1, 0, 0), (9, 50, 1, 0, 0),
        (1, 0, 0, 1, 0), (1, 0, 1, 1, 0), (1, 0, 0, 1, 256), (1, 0, 1, 1, 256)]


@pytest.mark.parametrize("G,nc,pb,grad,snap", ASKS)
def test_tail_plan_has_slots_and_tables_at_every_bin_count(rules, G, nc, pb, grad, snap):
    got = rules("plan_tail", [(n, G, nc, pb, grad, snap) for n in BINS])
    for n, g in zip(BINS, got):
        res, used = _tables(n, G, nc, pb, grad, snap)
        assert g[:6] == res, n
        slots = g[6]
        if n > 65_536:
            assert slots == 0
            continue
        assert slots == (64 if used + 64 * 8 * 80 <= 226 * KB else 32), n
        assert g[7] == used + slots * 8 * 80 <= 226 * KB


@pytest.mark.parametrize("G,nc,pb,grad,snap", ASKS)
@pytest.mark.parametrize("threads", [256, 512, 768, 1024])
@pytest.mark.parametrize("ext", [0, 1])
def test_main_plan_has_batches_and_tables_at_every_bin_count(rules, ext, threads, G, nc, pb, grad, snap):
    snap = threads if snap else 0
    got = rules("plan_main", [(threads, ext, n, G, nc, pb, grad, snap) for n in BINS])
    warps, rec = threads // 32, 1424 if ext else 1296
    for n, g in zip(BINS, got):
        res, used = _tables(n, G, nc, pb, grad, snap)
        assert g[:6] == res, n
        slots = g[6]
        if threads == 1024:
            assert slots == 0 and g[7] == used
            continue
        assert slots == (32 if used + warps * (48 + rec) <= 226 * KB else 16), n
        # two warps share a record of 32 slots where each has 16; the tables behind them are 16-byte aligned
        front = warps * 48 + warps * slots // 32 * rec
        assert front % 16 == 0 and g[7] == used + front <= 226 * KB
