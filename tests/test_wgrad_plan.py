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
extern "C" int nine(long long M, int cin, int cout, int Kp, int used, int per) {
    return lbm::nn::nine_taps_pay(M, cin, cout, Kp, used, per);
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


# one-tap / nine-tap, us a call, where one is faster by more than a fifth
@pytest.mark.parametrize("B,n,cin,cout,splits,one,nine", [
    (2, 64, 32, 32, 1, 1535, 2605), (2, 64, 32, 32, 8, 204, 364), (2, 64, 32, 32, 43, 115, 79), (2, 64, 32, 24, 4, 510, 924),
    (2, 64, 32, 24, 43, 133, 93), (2, 64, 64, 8, 8, 310, 482), (2, 64, 64, 8, 21, 324, 162), (2, 64, 96, 32, 4, 521, 688),
    (2, 64, 96, 32, 14, 251, 144), (4, 64, 96, 32, 32, 556, 208), (2, 64, 64, 64, 21, 172, 122), (4, 32, 64, 64, 2, 208, 396),
    (8, 32, 64, 16, 21, 119, 78), (4, 32, 256, 64, 5, 178, 121), (4, 32, 256, 64, 2, 273, 396), (2, 32, 128, 24, 1, 273, 487),
    (2, 32, 128, 24, 11, 84, 66), (2, 64, 128, 40, 4, 663, 924), (2, 64, 128, 40, 11, 664, 362), (1, 64, 32, 8, 4, 273, 480),
    (1, 64, 32, 8, 43, 109, 76), (1, 128, 32, 32, 16, 521, 688), (1, 128, 32, 32, 43, 345, 285), (1, 256, 32, 32, 8, 7613, 10202),
    (1, 256, 32, 32, 43, 2541, 1948), (1, 64, 256, 64, 1, 1010, 1335), (1, 64, 256, 64, 8, 375, 209)])
def test_the_form_is_the_faster_one(lib, B, n, cin, cout, splits, one, nine):
    M = B * n ** 3
    per = -(-(M // 64) // splits)
    lib.nine.argtypes = [ctypes.c_longlong] + [ctypes.c_int] * 5
    assert bool(lib.nine(M, cin, cout, (27 * cin + 63) // 64 * 64, -(-(M // 64) // per), per)) == (nine < one)
