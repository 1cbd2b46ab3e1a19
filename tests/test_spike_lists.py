"""Length of the spike-list ring (host build of the rule).

One sample with a readout delay keeps a ring longer than its update window,
so that its readout runs on the second stream, whatever gradient form its size
selects; rings of a gigabyte and batches keep the shortest ring that holds the
delayed list.
"""
from __future__ import annotations

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "spike_lists.h"
using namespace eprop;
int main() {
    const long long slot = 32 * 256 * 4;
    // (window, max delay, d_out, lists walked, batch, bytes per slot)
    printf("%d %d %d %d %d %d %d %d\n", spike_list_slots(300, 1, 2, false, 1, slot),
           spike_list_slots(300, 5, 0, false, 1, slot), spike_list_slots(300, 5, 0, true, 1, slot),
           spike_list_slots(300, 1, 7, false, 8, 8 * slot), spike_list_slots(1, 1, 64, true, 1, slot),
           spike_list_slots(1 << 20, 1, 3, false, 1, slot), spike_list_slots(20000, 1, 3, false, 1, slot),
           spike_list_slots(1 << 20, 1, 3, true, 1, slot));
}
"""


def test_ring_is_longer_than_the_window_where_the_readout_trails(tmp_path):
    (tmp_path / "l.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2511_21674_gb300", "csrc"),
                    str(tmp_path / "l.cpp"), "-o", str(tmp_path / "l")], check=True)
    out = subprocess.run([str(tmp_path / "l")], check=True, capture_output=True, text=True).stdout.split()
    assert [int(x) for x in out] == [302, 2, 306, 9, 66, 5, 20002, (1 << 20) + 2]
