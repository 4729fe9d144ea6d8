"""The slot order of the packed FP32 sweep's velocity groups (kgs::pack_order in
csrc/kgs_pack.h), compiled with the host C++ compiler: every velocity of a
group has one slot, in the half of the group that sums it; the slots of a
thread (2t and 2t + 1) within the paired part hold the same x node of two
neighbouring whole lines; the rest keep their order, so that a line's sums run
over its nodes as one line at a time would.
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
        for (int p : place) std::printf("%d ", p);
        std::printf("\n");
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def orders(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("pack")
    src, exe = d / "driver.cpp", d / "driver"
    src.write_text(DRIVER)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    ask = []
    for nxo in list(range(1, 41)) + [64, 127, 128, 129, 150, 300]:
        for lines in (1, 2, 3, 7, 16, 45, 121):
            total = nxo * lines
            ask += [(v0, min(256, total - v0), nxo) for v0 in range(0, total, 256)]
    text = "".join("%d %d %d\n" % a for a in ask)
    out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
    return list(zip(ask, [[int(x) for x in line.split()] for line in out.splitlines()]))


def test_pack_order(orders):
    assert len(orders) > 500
    for (v0, count, nxo), place in orders:
        assert sorted(place) == list(range(count)), (v0, count, nxo)
        for b in range(0, count, 128):
            half = place[b:b + 128]
            n = len(half)
            assert sorted(half) == list(range(b, b + n))
            head = min(n, -(v0 + b) % nxo)
            full = (n - head) // nxo
            paired = full // 2 * 2 * nxo
            for k in range(0, paired, 2):
                a, c = v0 + half[k], v0 + half[k + 1]
                assert a % nxo == c % nxo == k // 2 % nxo  # the same node, in node order
                assert c // nxo == a // nxo + 1            # neighbouring lines
                assert a // nxo == (v0 + b + head) // nxo + 2 * (k // (2 * nxo))
            assert half[paired:] == sorted(half[paired:])
