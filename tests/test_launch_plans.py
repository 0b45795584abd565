"""The launch plans of pf16_plan.h, compiled for the host on their own: the split-K
reduction's groups of splits for every split count the weight gradients take."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_1911_07384_gb300.build import CSRC

SHIM = """
#include "pf16_plan.h"
extern "C" void splitk(int splits, long long total, int* out) {
  const pf16::SplitkPlan p = pf16::splitk_plan(splits, total);
  out[0] = p.tree_groups_log2, out[1] = p.leaves_log2, out[2] = p.groups_log2, out[3] = p.leaf_step;
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plans")
    (d / "shim.cpp").write_text(SHIM)
    cxx = shutil.which("g++") or shutil.which("c++")
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "shim.so"),
                    str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(os.path.join(str(d), "shim.so"))


@pytest.mark.parametrize("total", [64, 96, 128, 256, 303, 304, 305, 512, 1152, 4096, 20000, 77823, 77824, 131072])
def test_splitk_groups(plans, total):
    """A CTA's 256 threads hold every group of a chunk, a thread at most 16 splits, and
    groups and splits per thread multiply to the padded split count."""
    out = (ctypes.c_int * 4)()
    for splits in list(range(1, 1025)) + [2048, 4096]:
        plans.splitk(splits, ctypes.c_longlong(total), out)
        tree, leaves, groups, step = out
        assert 0 <= groups <= 8 and 0 <= leaves <= 4, (splits, tuple(out))
        assert groups + leaves == (splits - 1).bit_length(), (splits, tuple(out))
        assert 0 <= tree <= 8 and tree <= groups + leaves, (splits, tuple(out))
        # a group lies inside a run of the tree, or is two single splits half of them apart
        if groups >= tree:
            assert step == 1
        else:
            assert leaves == 1 and groups + 1 == tree and step == 1 << groups
