"""Routes of the host code that one GPU cannot show, on a fake CUDA runtime
(no GPU needed)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_HOME = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def _run(tmp_path, cmd, exe):
    if not os.path.exists(os.path.join(CUDA_HOME, "include", "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.stdout, r.stderr)
    return r.stdout.splitlines()


def test_state_reads_from_another_current_device(tmp_path):
    """md_get_state copies by a kernel only when the handle's device is the
    current one (a launch on another device's stream fails) and owns the
    destination; otherwise by a copy, which needs neither."""
    gxx = shutil.which("g++") or pytest.skip("no C++ compiler")
    exe = str(tmp_path / "host_fakes")
    lines = _run(tmp_path, [gxx, "-std=c++17", "-O0", "-no-pie", os.path.join(ROOT, "tests", "c", "host_fakes.cpp"),
                            "-I", os.path.join(CUDA_HOME, "include"), "-o", exe, "-L",
                            os.path.join(CUDA_HOME, "lib64"), "-lcudart_static", "-lpthread", "-ldl", "-lrt",
                            "-Wl,--unresolved-symbols=ignore-all"], exe)
    assert lines == ["get_state current 0 owner 0: 0 kernel", "get_state current 0 owner 1: 0 copy",
                     "get_state current 1 owner 0: 0 copy", "get_state current 1 owner 1: 0 copy"]


def test_device_ordinals_past_the_cluster_table(tmp_path):
    """Devices from ordinal 64 on have no table of cluster slots: the cluster
    kernel's preparation succeeds there all the same, and every launch takes the
    persistent kernel."""
    nvcc = shutil.which("nvcc") or pytest.skip("no nvcc")
    exe = str(tmp_path / "device_ordinal")
    lines = _run(tmp_path, [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1",
                            "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"), "-o", exe,
                            os.path.join(ROOT, "tests", "c", "device_ordinal.cu")], exe)
    assert lines == [f"device {d}: 0, 0" for d in (64, 127, 500)]
