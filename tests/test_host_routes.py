"""Routes of the host code that one GPU cannot show, on a fake CUDA runtime
(no GPU needed)."""
import os
import shutil
import subprocess

import pytest

from tests.attention_shapes import CLUSTER, NOALLOC_PERSISTENT

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_HOME = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def _run(cmd, exe, text=""):
    if not os.path.exists(os.path.join(CUDA_HOME, "include", "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60, input=text)
    assert r.returncode == 0, (r.stdout, r.stderr)
    return r.stdout.splitlines()


def test_state_reads_from_another_current_device(tmp_path):
    """md_get_state copies by a kernel only when the handle's device is the
    current one (a launch on another device's stream fails) and owns the
    destination; otherwise by a copy, which needs neither."""
    gxx = shutil.which("g++") or pytest.skip("no C++ compiler")
    exe = str(tmp_path / "host_fakes")
    lines = _run([gxx, "-std=c++17", "-O0", "-no-pie", os.path.join(ROOT, "tests", "c", "host_fakes.cpp"),
                            "-I", os.path.join(CUDA_HOME, "include"), "-o", exe, "-L",
                            os.path.join(CUDA_HOME, "lib64"), "-lcudart_static", "-lpthread", "-ldl", "-lrt",
                            "-Wl,--unresolved-symbols=ignore-all"], exe)
    assert lines == ["get_state current 0 owner 0: 0 kernel", "get_state current 0 owner 1: 0 copy",
                     "get_state current 1 owner 0: 0 copy", "get_state current 1 owner 1: 0 copy"]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    """Runs the cluster kernel's host code on the given lines."""
    nvcc = shutil.which("nvcc") or pytest.skip("no nvcc")
    exe = str(tmp_path_factory.mktemp("rule") / "cluster_rule")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-I",
           os.path.join(ROOT, "include"), "-o", exe, os.path.join(ROOT, "tests", "c", "cluster_rule.cu")]
    _run(cmd, exe)
    return lambda text: _run(["true"], exe, text)


def test_device_ordinals_past_the_cluster_table(rule):
    """Devices from ordinal 64 on have no table of cluster slots: the cluster
    kernel's preparation succeeds there all the same, and every launch takes the
    persistent kernel."""
    assert rule("") == [f"device {d}: 0, 0" for d in (64, 127, 500)]


def test_the_shapes_of_the_gpu_tests_take_their_kernels(rule):
    """On a GB300 the cost rule takes, for the shapes the GPU tests list, the form
    (or the persistent kernel) that they are listed for."""
    ask, want = [], []
    for (L, Hq, Hkv, ps, lengths, aligned), form in CLUSTER:
        if form:     # the step's new token is on its page when the rule decides
            n = [x + 1 for x in lengths]
            scratch = 512 * 2 * 8 * min(4096, (max(n) + ps - 1) // ps * ps)
            ask.append([L, Hkv, ps, scratch, len(n), *n])
            want.append("form %d %d %d" % form)
    for L, Hq, Hkv, ps, lengths in NOALLOC_PERSISTENT:
        ask.append([L, Hkv, ps, 0, len(lengths), *lengths])
        want.append("form 0 4 0")
    got = rule("\n".join(" ".join(map(str, a)) for a in ask) + "\n")
    assert got[3:] == want
