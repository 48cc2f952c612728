"""Which runs of steps lbm_step launches as graphs (csrc/run_lengths.h), compiled for the host: how
many graphs a sequence of runs makes, and which of its runs go as graphs."""
import ctypes
import os
import subprocess

import pytest

import paper_1710_04751_gb300

HEADER = os.path.join(os.path.dirname(paper_1710_04751_gb300.__file__), "csrc", "run_lengths.h")
SOURCE = """
#include "%s"
// made: lengths that were given a slot; graphed: runs that found one; busy: the stream is never idle
extern "C" void drive(const long long* runs, int count, int busy, int fail_at, int* made, int* graphed) {
    lbm::RunLengths r;
    *made = *graphed = 0;
    for (int i = 0; i < count; ++i) {
        if (i == fail_at) r.failed = true;
        bool replaced;
        const int slot = r.find(runs[i], &replaced);
        if (slot < 0) continue;
        if (slot >= lbm::RunLengths::kSlots) *made = -1000;
        if (replaced && busy && r.len[slot]) continue;
        if (replaced) r.take(slot, runs[i]), ++*made;
        ++*graphed;
    }
}
""" % HEADER


@pytest.fixture(scope="module")
def drive(tmp_path_factory):
    d = tmp_path_factory.mktemp("runs")
    (d / "runs.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-o", str(d / "runs.so"), str(d / "runs.cpp")],
                   check=True)
    L = ctypes.CDLL(str(d / "runs.so"))

    def call(runs, busy=0, fail_at=-1):
        made, graphed = ctypes.c_int(), ctypes.c_int()
        L.drive((ctypes.c_longlong * len(runs))(*runs), len(runs), busy, fail_at, ctypes.byref(made), ctypes.byref(graphed))
        return made.value, graphed.value
    return call


@pytest.mark.parametrize("busy", [0, 1])
@pytest.mark.parametrize("runs,made,graphed", [
    ([10] * 50, 1, 49),
    ([10, 10, 20, 20] * 50, 2, 198),
    ([10, 10, 20, 20, 30, 30] * 50, 2, 198),  # a third length in pairs displaces none
    ([10, 10, 20, 20, 10, 20, 10, 20], 2, 6),
    ([10, 20, 30] * 50, 0, 0),
    ([3] * 50 + [129] * 50 + [0, 0], 0, 0),
    (list(range(4, 129)), 0, 0)])
def test_graphs_that_a_sequence_of_runs_makes(drive, runs, made, graphed, busy):
    assert drive(runs, busy) == (made, graphed)


def test_a_length_that_stays_displaces_the_one_used_less_recently(drive):
    pairs = [10, 10, 20, 20]
    # 30 is launched step by step 15 times, then displaces 10: 20 keeps its graphs, 10 has to come 16 times
    assert drive(pairs + [30] * 40) == (3, 2 + 25)
    assert drive(pairs + [30] * 40 + [20] * 3) == (3, 2 + 25 + 3)
    assert drive(pairs + [30] * 40 + [10] * 15) == (3, 2 + 25)
    assert drive(pairs + [30] * 40, busy=1) == (2, 2)


def test_no_graph_after_a_failure(drive):
    assert drive([10] * 50, fail_at=20) == (1, 19)
