"""The rules by which rows and groups are shared by clusters of CTAs, compiled for the host: no cluster wider than the device can
place is ever asked for (a partition of a GPU may have no 16 SMs in one GPC), and none that another rule would cut."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2607_11976_b200 import build

SOURCE = """
#include "lt_cluster_width.h"
extern "C" int select_width(int n_keys, int n_rows, int widest) { return lt::select_cluster_width(n_keys, n_rows, widest); }
extern "C" int union_width(int n_groups, int rows, long long entries, int sms, int ctas_at_once, int widest) {
  return lt::union_cluster_width(n_groups, rows, entries, sms, [&](int w) { return w > widest ? 0 : ctas_at_once / w; });
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SOURCE)
    out = os.path.join(d, "rules.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-o", out, str(d / "rules.cpp")], check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("widest", [1, 2, 4, 8, 16])
def test_select_never_asks_for_more_than_the_device_places(rules, widest):
    for n_keys in (16385, 32768, 32769, 65537, 131072, 131073, 1 << 20, 2 ** 31 - 1):
        for n_rows in (1, 8, 9, 148, 1 << 20, 2 ** 31 - 1):
            width = rules.select_width(n_keys, n_rows, widest)
            assert 1 <= width <= widest and width & (width - 1) == 0
            assert width <= 8 or n_rows * width <= 128
    wide = rules.select_width(131073, 8, widest)
    assert wide == widest


def test_select_widths_at_measured_points(rules):
    """(keys, rows) -> the width that measured best; below, both sides of the line between shares of 8192 and of 16384 keys (32 CTAs of the
    row count times the width before it is doubled) and of the widths beyond which a share is never short."""
    for n_keys, n_rows, best in ((20000, 1, 4), (40000, 7, 8), (131072, 1, 8), (131073, 8, 16), (131073, 9, 8)):
        assert rules.select_width(n_keys, n_rows, 16) == best
    for n_keys, n_rows, width in ((16385, 16, 4), (16385, 17, 2), (32768, 8, 4), (32769, 8, 8), (32769, 9, 4), (32768, 17, 2), (65536, 8, 8), (65536, 9, 4),
                                  (65537, 9, 8), (131072, 2, 8)):
        assert rules.select_width(n_keys, n_rows, 16) == width


@pytest.mark.parametrize("widest", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("ctas_at_once", [16, 148, 592])
def test_union_runs_in_one_wave(rules, widest, ctas_at_once):
    for n_groups in (1, 2, 8, 16, 64, 125, 592, 4096):
        for rows, topk in ((1, 1), (2, 4096), (8, 32), (16, 512), (64, 2048), (4096, 4096)):
            width = rules.union_width(n_groups, rows, ctypes.c_longlong(rows * topk), 148, ctas_at_once, widest)
            assert 1 <= width <= min(widest, 2 * rows - 1) and width & (width - 1) == 0
            if width > 1:
                assert n_groups * width <= ctas_at_once and rows * topk // width >= 256
                assert width <= 8 or n_groups * width <= 128


def test_union_widths_at_measured_points(rules):
    """(groups, rows, topk, CTAs of that shared memory an SM holds) -> the width that measured best."""
    for n_groups, rows, topk, per_sm, best in ((64, 64, 2048, 4, 8), (64, 64, 2048, 2, 4), (64, 16, 512, 2, 2), (128, 8, 32, 2, 1),
                                               (125, 4, 1024, 4, 1), (64, 64, 2048, 1, 2), (1, 64, 2048, 4, 16), (32, 128, 512, 4, 8), (32, 32, 2048, 3, 8)):
        assert rules.union_width(n_groups, rows, ctypes.c_longlong(rows * topk), 148, 148 * per_sm, 16) == best
