"""Checks of the fixed-point kernels' code that need no GPU: tests/c/fx_host.cu, compiled with
nvcc and run on the host."""
import os
import subprocess

import pytest

from paper_1501_04438_gb300 import build as gsm_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def compile_host(tmp, name):
    """tests/c/<name>.cu as a host program."""
    try:
        nvcc = gsm_build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = str(tmp / name)
    subprocess.run([nvcc, *gsm_build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", gsm_build.CSRC,
                    os.path.join(ROOT, "tests", "c", name + ".cu"), "-o", exe], check=True)
    return exe


def test_sync_groups_of_the_64r_kernels_have_words_of_their_own(tmp_path):
    """The sync groups of a CTA are ordered by barriers of their own only, so no two may use the same
    word of the shared reduction arrays."""
    out = subprocess.run([compile_host(tmp_path, "fx_host")], check=True, capture_output=True, text=True).stdout
    assert out.split() == ["0"] * 7


def test_multiplied_lines_are_no_worse_than_in_doubles(tmp_path):
    """Maximum error of one multiplied line (smooth, a point, white noise, a wave near Nyquist, a point
    over a floor, alternating; short and long lines) at most that of a plain FFT in doubles."""
    out = subprocess.run([compile_host(tmp_path, "fx_accuracy")], check=True, capture_output=True, text=True).stdout
    lines = [line.split() for line in out.splitlines()]
    assert len(lines) == 36
    assert not [line for line in lines if float(line[2]) > float(line[3])], out
