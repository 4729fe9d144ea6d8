"""Choices of the autotuner kept in a file (KGS_AUTOTUNE_CACHE): one timed on
other kernels, whose key carries another revision or none, is not taken.
Needs no GPU: a choice in the file is returned before any timing.
"""
import re

import pytest

from paper_1810_00348_gb300 import inputs, kgs


def tune(p):
    """The shape, or None where it would have to be timed and cannot be (no GPU)."""
    try:
        return kgs.kgs_autotune(p, precision=kgs.KGS_MIXED)
    except kgs.KgsError:
        return None


def revision():
    src = open(kgs.HERE + "/csrc/kgs_autotune.cu").read()
    return int(re.search(r"KERNEL_REVISION = (\d+);", src).group(1))


@pytest.mark.parametrize("mark,taken", [("", False), ("r%d_" % (revision() - 1), False), ("r%d_" % revision(), True)])
def test_only_choices_of_this_revision_are_taken(tmp_path, monkeypatch, mark, taken):
    n = 5 + len(mark) + taken  # a size of its own: the process remembers every choice
    p = inputs.cavity([n, 6, 7], [5, 4, 3], Kn=0.5)
    path = tmp_path / "shapes"
    path.write_text("%sp1_c%dx6x7_v5x4x3_s0 256 12 0.100000\n" % (mark, n))  # 12: never a candidate
    monkeypatch.setenv("KGS_AUTOTUNE_CACHE", str(path))
    assert (tune(p) == (256, 12)) == taken
