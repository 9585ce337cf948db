"""Warp-level device code run lane by lane on the host under a race detector: lanes
may pass data through memory only across __syncwarp (shuffles and votes order
nothing in the programming model)."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2308_11892_gb300", "csrc")


def _run(tmp_path, source, *args):
    flags = ["-std=c++17", "-O1", "-g", "-ffp-contract=off", "-w", "-pthread",
             "-fsanitize=thread"]
    probe = tmp_path / "probe.cpp"
    probe.write_text("int main() { return 0; }\n")
    pexe = str(tmp_path / "probe")
    r = subprocess.run(["g++", *flags, str(probe), "-o", pexe], capture_output=True)
    if r.returncode or subprocess.run([pexe], capture_output=True).returncode:
        pytest.skip("no usable thread sanitizer")
    exe = str(tmp_path / "lanes")
    dirs = [f"-I{d}" for d in (os.path.join(HERE, "lane_order"), CSRC, tmp_path)]
    subprocess.run(["g++", *flags, *dirs, os.path.join(HERE, "lane_order", source), "-o", exe],
                   check=True)
    env = dict(os.environ, TSAN_OPTIONS="exitcode=66 halt_on_error=1")
    r = subprocess.run([exe, *args], capture_output=True, text=True, timeout=600, env=env)
    assert r.returncode == 0, (r.stdout + r.stderr)[-3000:]


def test_product_accumulators(tmp_path):
    _run(tmp_path, "products.cpp")


def test_interpolation_by_lane_groups(tmp_path):
    _run(tmp_path, "interp.cpp")


def _ilu_kernel(tmp_path):
    """k_ilu_factor_pair with what it calls, cut from setup_ilu.cu."""
    src = open(os.path.join(CSRC, "setup_ilu.cu")).read()
    inv = src[src.index("__device__ __forceinline__ double inv4_pair"):]
    row = src[src.index("constexpr int kRowMax"):src.index("__global__ void k_max_row")]
    (tmp_path / "ilu_pair.inc").write_text(inv[:inv.index("\n}\n") + 3] + row)


def test_ilu_two_rows_per_warp(tmp_path):
    _ilu_kernel(tmp_path)
    _run(tmp_path, "ilu.cpp")


def test_ilu_two_rows_per_warp_rounds_as_the_definition(tmp_path):
    _ilu_kernel(tmp_path)
    _run(tmp_path, "ilu.cpp", "bits")
