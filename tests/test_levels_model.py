"""The level arithmetic of the compact latent state against the entry-by-entry update, on the CPU:
levels_host.cu compiles the same header for the host and walks random moves over random thresholds
(uniform, decades apart, tiny, repeated and zero), comparing every sum and every entry exactly."""
import pathlib
import subprocess

import pytest

from paper_2210_04184_gb300 import build as _build

HERE = pathlib.Path(__file__).resolve().parent


def test_levels_equal_the_entries(tmp_path):
    try:
        nvcc = _build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    exe = tmp_path / "levels_host"
    subprocess.run([nvcc, _build.ARCH, "-O2", "-std=c++17", f"-I{_build.CSRC}", str(HERE / "levels_host.cu"), "-o",
                    str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout
