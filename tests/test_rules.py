"""The launch rules (csrc/rules.h) that are plain arithmetic, built by the host compiler.

* a round of the tail's events always goes on, up to the last event number.
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
int main(int argc, char** argv) {
  // round_end <e> <span> <max_events> ...
  for (int i = 1; i + 3 < argc; i += 4)
    if (!strcmp(argv[i], "round_end"))
      printf("%u\n", round_end(strtoul(argv[i + 1], 0, 0), strtoul(argv[i + 2], 0, 0), strtoul(argv[i + 3], 0, 0)));
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

    def call(*args):
        out = subprocess.run([str(exe), *map(str, args)], check=True, capture_output=True, text=True).stdout
        return [[int(x) for x in line.split()] for line in out.splitlines()]
    return call


@pytest.mark.parametrize("max_events", [1, 2, 64, 777, 2 ** 31, 2 ** 32 - 64, 2 ** 32 - 2, 2 ** 32 - 1])
@pytest.mark.parametrize("span", [1, 2, 32, 64, 65536])
def test_tail_rounds_go_on_to_the_last_event(rules, span, max_events):
    last = max_events - 1
    starts = sorted({e for e in (0, 1, last - 2 * span, last - span - 1, last - span, last - span + 1, last - 2,
                                 last - 1, last) if 0 <= e <= last})
    got = rules(*[a for e in starts for a in ("round_end", e, span, max_events)])
    for e, (end,) in zip(starts, got):
        assert end == min(e + span, last)
        assert end > e or e == last
