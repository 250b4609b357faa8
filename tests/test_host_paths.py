"""The library's host code on the CPU, with a fake of the CUDA runtime in which
calls can be made to fail: paths that a healthy GPU does not take."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

from paper_1812_05401_gb300 import build as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TESTS_C = os.path.join(ROOT, "tests", "c")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    B.build()
    objs = [os.path.join(B.BUILD, src.replace(".cu", ".o")) for src in B.SOURCES]
    if not all(map(os.path.exists, objs)):
        B.build(force=True)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(B._nvcc())))), "include")
    exe = str(tmp_path_factory.mktemp("host") / "host_paths")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", cuda, "-I", os.path.join(ROOT, "include"), "-I", B.CSRC,
                    os.path.join(TESTS_C, "host_paths.cpp"), *objs, "-o", exe, "-ldl", "-lpthread"], check=True)
    return exe


def _run(program, path):
    r = subprocess.run([program, path], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("path", ["failed_call", "failed_call_vector", "failed_call_pairs", "failed_sum"])
def test_failed_calls_keep_the_records_of_their_steps(program, path):
    """One node per thread, a vector of nodes per thread, and two steps a launch."""
    _run(program, path)


def test_captured_pairs_swap_buffers_as_single_steps(program):
    _run(program, "captured_pairs")


@pytest.mark.parametrize("path", ["second_mask", "second_mask_refused"])
def test_second_mask_is_taken_by_the_first_pair(program, path):
    _run(program, path)


@pytest.mark.parametrize("path", ["refused_window", "refused_mask"])
def test_refused_buffers_leave_no_error(program, path):
    _run(program, path)


@pytest.mark.parametrize("path", ["window_f64", "window_f64_mid", "window_f32", "window_f16"])
def test_record_windows_are_bounded(program, path):
    _run(program, path)


def test_grouped_calls_copy_their_tables_at_once(program):
    _run(program, "grouped_tables")


def test_the_step_kernel_has_its_name(program):
    _run(program, "named_kernel")
