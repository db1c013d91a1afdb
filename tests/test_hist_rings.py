"""The histogram's shared-memory rings (one CTA per SM) at every block size a
context may have: the kernel's own arithmetic (lk_layout.h), compiled for the
host.  Each warp's ring starts on a 16-byte boundary (it is the destination of
bulk copies and of 128-bit reads), holds whole vectors, and meets neither
another ring, the counter table nor the end of the shared memory."""
import shutil
import subprocess

import pytest

from paper_2310_01212_gb300 import build

SOURCE = r"""
#include <stdio.h>
#include "lk_layout.h"
int main() {
  /* the table's offset: what is left to a 64 KB boundary of the shared window */
  for (uint32_t dsm = 1024; dsm <= 32768; dsm += 128)
    for (uint32_t w = 2; w <= 32; ++w)
      for (uint32_t i = 0; i < w; ++i) {
        const uint32_t tbl = 65536u - dsm, off = lk_hist_ring_off(w, i, tbl);
        printf("%u %u %u %u %u %u\n", w, i, dsm, tbl, off, lk_hist_stage_vecs(w) * LK_STAGES * 16u);
      }
  printf("smem %u table %u\n", LK_TC_SMEM, LK_HIST_TABLE);
}
"""


def test_rings_at_every_block_size(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "rings.cpp", str(tmp_path / "rings")
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", f"-I{build.CSRC}", str(src), "-o", exe], check=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()
    smem, table = (int(x) for x in lines.pop().split()[1::2])
    assert len(lines) == sum(range(2, 33)) * len(range(1024, 32768 + 1, 128))
    taken = {}
    for line in lines:
        w, i, dsm, tbl, off, size = (int(x) for x in line.split())
        assert (dsm + off) % 16 == 0 and size % 16 == 0, (32 * w, i, off)
        assert size >= 4 * 16 * 32, (32 * w, size)              # at least a vector a lane in every stage
        assert 0 <= off and off + size <= smem, (32 * w, i, off)
        taken.setdefault((w, dsm), [(tbl, tbl + table)]).append((off, off + size))
    for (w, _), spans in taken.items():
        spans.sort()
        assert len(spans) == w + 1
        assert all(a[1] <= b[0] for a, b in zip(spans, spans[1:])), (32 * w, spans)
