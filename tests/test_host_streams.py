"""Host code of the C entry points (csrc/kvs_api.cu) on a CUDA runtime that runs nothing (fake_cuda.cpp): which stream does what, in
which order, on which memory."""
import os
import subprocess

import pytest

from paper_2601_22996_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fake") / "host_streams")
    subprocess.check_call([os.environ.get("NVCC", "nvcc"), "-x", "c++", "-std=c++17", "-O2", "-cudart", "none", "-I", build._INCLUDE, "-I", build._CSRC,
                           os.path.join(HERE, "fake_cuda.cpp"), os.path.join(build._CSRC, "kvs_api.cu"), "-o", exe])
    return exe


def _run(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


def test_chunks_of_the_host_entry_point_share_no_scratch(program):
    """Chunks of unequal size or composition take turns on the lanes: no kernel uses scratch, results or inputs that another
    one, not ordered before or after it, writes."""
    _run(program, "overlaps")


def test_failures_leave_nothing_in_flight(program):
    """A refused call launches nothing; after one that fails at any point (a runtime call, a launch, host memory), no kernel and no
    copy of it is left for the next call to race with, and no exception leaves the C entry point."""
    _run(program, "errors")


def test_requests_for_sizes_belong_to_their_reader(program):
    """Requests that overlap each get their own sizes; one reader refuses a second request; page-locked memory is neither overwritten nor
    given back while a copy uses it."""
    _run(program, "sizes")


def test_groups_of_speculative_evaluations(program):
    """One, two, five and eight budgets per instance, few evaluations and many: a CTA has room for what its group holds, groups are of near-equal
    size, an SM has as many evaluations in flight as it can hold, and the kernel in memory takes over where it is the faster one."""
    _run(program, "groups")
