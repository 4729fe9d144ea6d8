"""The units in which the moment phase of the packed FP32 sweep sums a half of
a velocity group (kgs::PackHalf in csrc/kgs_pack.h), compiled with the host C++
compiler: walking the units as the kernel does, every slot of kgs::pack_order
must meet the line and the x node of the velocity that it holds, also where
the half lies inside one line and its first unit ends before the line does.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1810_00348_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "kgs_pack.h"
int main()
{
    int v0, count, nxo;
    std::vector<int> place;
    while (std::scanf("%d %d %d", &v0, &count, &nxo) == 3) {
        kgs::pack_order(v0, count, nxo, place);
        int bad = 0, seen = 0;
        auto meet = [&](int slot, int line, int node) {
            seen++;
            bad += slot >= count || v0 + place[slot] != line * nxo + node;
        };
        for (int mb = 0; mb < count; mb += kgs::PACK_HALF) {
            const kgs::PackHalf h(v0 + mb, std::min(kgs::PACK_HALF, count - mb), nxo);
            const int pairs = h.full / 2, units = (h.head > 0) + pairs + (h.full & 1) + (h.tail > 0);
            int line = (v0 + mb) / nxo, seq = mb + 2 * pairs * nxo;
            for (int u = 0; u < units; u++) {
                const int k = u - (h.head > 0);
                if (k >= 0 && k < pairs) {
                    for (int ix = 0; ix < nxo; ix++)
                        for (int l = 0; l < 2; l++) meet(mb + 2 * (k * nxo + ix) + l, line + l, ix);
                    line += 2;
                } else {
                    const int n = k < 0 ? h.head : (k == pairs && (h.full & 1)) ? nxo : h.tail;
                    const int ix0 = k < 0 ? h.first : 0;
                    for (int ix = ix0; ix < ix0 + n; ix++) meet(seq++, line, ix);
                    line++;
                }
            }
        }
        std::printf("%d %d\n", bad, seen - count);
    }
    return 0;
}
"""


def test_units_meet_the_velocity_of_every_slot(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "driver.cpp", tmp_path / "driver"
    src.write_text(DRIVER)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    ask = []
    for nxo in list(range(1, 41)) + [64, 127, 128, 129, 130, 133, 150, 200, 257, 260, 300]:
        for lines in (1, 2, 3, 6, 7, 16, 45):
            total = nxo * lines
            ask += [(v0, min(256, total - v0), nxo) for v0 in range(0, total, 256)]
    text = "".join("%d %d %d\n" % a for a in ask)
    out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
    assert len(out) == len(ask)
    wrong = [a for a, line in zip(ask, out) if line != "0 0"]
    assert not wrong, "%d groups, the first (v0, count, nxo): %s" % (len(wrong), wrong[:5])
