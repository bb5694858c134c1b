"""Host code of the library against a CUDA runtime on the host
(host_runtime/fake_cudart.cpp): allocations that fail in turn, and streams that
run as late as the runtime's documentation allows.  No GPU takes part."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host_runtime")


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    from paper_2203_10000_gb300 import build
    build.build()
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
    exe = str(tmp_path_factory.mktemp("host_runtime") / "driver")
    objs = [os.path.join(build.BUILD, s + ".o") for s in build.SOURCES]
    inc = ["-I", os.path.join(cuda, "include"), "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include")]
    r = subprocess.run(["g++", "-std=c++17", "-O1", *inc, os.path.join(HERE, "driver.cpp"),
                        os.path.join(HERE, "fake_cudart.cpp"), *objs, "-ldl", "-lpthread", "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    return exe


def _run(driver, scenario):
    r = subprocess.run([driver, scenario], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]


def test_failed_allocations_leave_the_context_usable(driver):
    _run(driver, "out_of_memory")


def test_uploads_are_ordered_with_the_kernels_that_read_them(driver):
    _run(driver, "uploads")


def test_a_recorded_error_is_reported_once(driver):
    _run(driver, "status_once")


def test_host_meshes_without_tets_keep_their_nodes(driver):
    _run(driver, "no_tets")


def test_anchors_cut_short_make_no_grid(driver):
    _run(driver, "anchors_cut_short")


def test_large_construction_scratch_is_given_back(driver):
    _run(driver, "scratch_given_back")


def test_a_priority_order_uploads_its_rows(driver):
    _run(driver, "priority_uploads")


def test_cell_lists_beyond_32_bits_make_no_grid(driver):
    _run(driver, "sums_beyond_32_bits")


def test_lists_are_cleared_after_a_failed_call(driver):
    _run(driver, "lists_cleared_after_a_failure")


def test_long_thin_triangles_do_not_fill_the_registration(driver):
    _run(driver, "needles")


def test_small_host_calls_without_page_locked_memory(driver):
    _run(driver, "no_pinned_memory")
