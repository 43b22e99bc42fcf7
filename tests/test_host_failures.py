"""CPU: the library's host code where device memory runs short, and what it asks
of the runtime.  The
library's objects are linked with a stand-in for the CUDA runtime
(tests/native/fake_cuda.cpp) that needs no GPU and fails allocations on demand."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def objects():
    from paper_2601_21990_gb300 import _build

    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("nvcc not available")
    _build.build()
    objs = [os.path.join(_build.BUILD, s.replace(".cu", ".o")) for s in _build.SOURCES]
    newest = max(os.path.getmtime(f) for f in _build._deps())
    if not all(os.path.exists(o) and os.path.getmtime(o) >= newest for o in objs):
        _build.build(force=True)
    return objs


def _run(objects, tmp_path, name):
    from paper_2601_21990_gb300 import _build

    exe = tmp_path / name
    subprocess.check_call([_build.nvcc(), *_build.ARCH, "-O1", "-std=c++17", "-cudart", "none", "-I", _build.INCLUDE,
                           "-I", _build.CSRC, os.path.join(ROOT, "tests", "native", name + ".cu"),
                           os.path.join(ROOT, "tests", "native", "fake_cuda.cpp"), *objects, "-lpthread",
                           "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip().endswith("ok"), out.stdout[-2000:] + out.stderr[-2000:]


def test_a_threshold_change_without_memory_keeps_the_rows(objects, tmp_path):
    _run(objects, tmp_path, "set_tuning_alloc_test")


def test_a_layout_without_memory_leaves_the_step_kernels(objects, tmp_path):
    _run(objects, tmp_path, "resident_alloc_test")


def test_a_servers_budget_covers_layouts_and_requests_come_first(objects, tmp_path):
    _run(objects, tmp_path, "serve_layout_test")


def test_admission_takes_as_many_calls_for_any_number_of_infeasible_lps(objects, tmp_path):
    _run(objects, tmp_path, "admit_calls_test")
