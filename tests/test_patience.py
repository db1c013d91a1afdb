"""The time limit of a wait for a CTA that may be several descriptors behind
(finite lists whose CTAs read the ring themselves): the rule itself
(lk_layout.h), compiled for the host.  The wait goes on while the cluster
finishes descriptors and runs out one limit after it stopped."""
import shutil
import subprocess

import pytest

from paper_2310_01212_gb300 import build

SOURCE = r"""
#include <stdio.h>
#include "lk_layout.h"
/* a wait from t = 1000 with this limit, checked every 10 ns, of a cluster that
 * finishes a descriptor every `every` ns until `stop`: when does it give up? */
static uint64_t gives_up(uint64_t limit, uint64_t every, uint64_t stop, uint64_t end) {
  lk_patience p = {0, 1000 + limit};
  for (uint64_t t = 1010; t < end; t += 10) {
    const uint64_t moving = t < stop ? t : stop;
    if (lk_out_of_patience(&p, t, moving / every, limit)) return t;
  }
  return 0;
}
int main() {
  printf("%llu\n", (unsigned long long)gives_up(2000, 1ull << 40, 0, 100000));       /* never moves */
  printf("%llu\n", (unsigned long long)gives_up(2000, 1500, 50000, 40000));          /* moves all along */
  printf("%llu\n", (unsigned long long)gives_up(2000, 1500, 9000, 100000));          /* moves, then stops */
  printf("%llu\n", (unsigned long long)gives_up(2000, 5000, 1ull << 40, 100000));    /* too slow */
}
"""


def test_the_limit_counts_from_the_last_progress(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "patience.cpp", str(tmp_path / "patience")
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", f"-I{build.CSRC}", str(src), "-o", exe], check=True)
    never, moving, stopped, slow = (int(x) for x in subprocess.run([exe], check=True, capture_output=True,
                                                                   text=True).stdout.split())
    assert 3000 < never <= 3010
    assert moving == 0
    assert 11000 < stopped <= 11010        # the last change, at t = 9000, and the limit
    assert 3000 < slow <= 3010             # gave up before the first change at t = 5000
