"""How the nine-tap weight gradient splits its voxels (csrc/nn/wgrad_plan.h), compiled for the host."""
import ctypes
import os
import subprocess

import pytest

import paper_1710_04751_gb300

HEADER = os.path.join(os.path.dirname(paper_1710_04751_gb300.__file__), "csrc", "nn", "wgrad_plan.h")
SOURCE = """
#include "%s"
extern "C" void plan(int total, int cin, int cout, int max_slices, int* out) {
    const lbm::nn::Wgrad9Plan p = lbm::nn::plan_wgrad9(total, cin, cout, max_slices);
    out[0] = p.slices, out[1] = p.ctas, out[2] = p.per;
}
""" % HEADER


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-o", str(d / "plan.so"), str(d / "plan.cpp")],
                   check=True)
    return ctypes.CDLL(str(d / "plan.so"))


# blocks of 64 voxels: batches of 16^3 to 256^3 grids
@pytest.mark.parametrize("total", [64, 320, 512, 1088, 4096, 8192, 12288, 16384, 32768, 65536, 262144])
def test_no_chain_is_longer_than_the_callers_split_makes_it(lib, total):
    out = (ctypes.c_int * 3)()
    for cin in (32, 64, 96, 128, 160, 256, 512):
        for cout in (8, 32, 40, 64):
            for splits in list(range(1, 64)) + [128, 304, total, total + 5]:
                chain = -(-total // splits)
                used = -(-total // chain)  # the slices the caller's workspace holds
                lib.plan(total, cin, cout, used, out)
                slices, ctas, per = out
                assert per <= chain, (cin, cout, splits)
                assert 1 <= slices <= used and ctas in (1, 2)
                assert slices * ctas * per >= total > (slices * ctas - ctas) * per
