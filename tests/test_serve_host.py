"""The server's batcher with the solver replaced by fakes, on the host: what a request
gets when a batched solve, or one system of it, does not end well."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    return inc


def _run(tmp_path, mode):
    csrc = os.path.join(ROOT, "paper_2308_11892_gb300", "csrc")
    shutil.copy(os.path.join(csrc, "serve.cu"), tmp_path / "serve.cpp")
    exe = str(tmp_path / "batches")
    dirs = [str(tmp_path), csrc, os.path.join(ROOT, "include"), _cuda_include()]
    subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-w", "-pthread", "-fsanitize=address",
                    *[f"-I{d}" for d in dirs],
                    os.path.join(HERE, "serve_host", "batches.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe, mode], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.stdout + r.stderr)[-3000:]


def test_failed_batch_keeps_its_message(tmp_path):
    """Every request of a batch that fails as a whole reports it; the message is read
    while the context that holds it exists."""
    _run(tmp_path, "fail")


def test_timed_out_system_fails_alone(tmp_path):
    """A system whose wait gave up, like one that broke down, leaves the other requests
    of its batch their results."""
    _run(tmp_path, "timeout")
