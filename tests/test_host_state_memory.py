"""The memory of a context's states, run on a fake of the CUDA runtime (tests/host) whose allocations
can fail: the library's host code as it is, no GPU."""
import os
import subprocess

import pytest

from paper_2601_00705_gb300 import build

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    out = tmp_path_factory.mktemp("host")
    flags = [*build.ARCH_FLAGS, "-O1", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC]
    sources = (os.path.join(build.CSRC, "rgs_api.cu"), os.path.join(HOST, "state_memory.cu"),
               os.path.join(HOST, "fake_runtime.cpp"))
    objects = []
    for src in sources:
        objects.append(str(out / (os.path.basename(src) + ".o")))
        subprocess.run([build.nvcc_path(), *flags, "-c", src, "-o", objects[-1]], check=True)
    exe = str(out / "state_memory")
    subprocess.run([build.nvcc_path(), "-cudart", "none", *objects, "-o", exe], check=True)
    return exe


def _run(program, name):
    r = subprocess.run([program, name], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-500:]


def test_a_forward_that_runs_out_of_memory_leaves_nothing_stale(program):
    _run(program, "failed_growth")


def test_a_first_forward_that_fails_leaves_no_state(program):
    _run(program, "failed_first")


def test_every_allocation_frees_the_kept_states_before_it_fails(program):
    _run(program, "kept_states_give_way")


def test_lists_past_the_blends_positions_are_refused(program):
    _run(program, "list_limits")


def test_reserved_pairs_take_their_documented_memory_and_serve_captures(program):
    _run(program, "reserved_pairs")


def test_kept_memory_is_bounded_and_given_back(program):
    _run(program, "kept_memory")


def test_a_reserve_between_a_forward_and_its_backward_keeps_the_pairs(program):
    _run(program, "reserve_after_forward")
