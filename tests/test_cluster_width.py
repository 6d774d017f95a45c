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
