"""CPU: the staged FFTs of the general lengths (shf_gfft.cuh), compiled for the
host and run item by item for every length 2^a 3^b 5^c up to 2048 against FP64
DFTs.  The bound 4 eps log2 L of the outputs' root mean square allows about four
rounding errors (eps = 6e-8) per factor of two."""

import os
import subprocess

import pytest

from paper_1112_1805_gb300 import build as nbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_general_lengths_match_the_dft(tmp_path):
    try:
        nvcc = nbuild.nvcc_path()
    except RuntimeError as e:
        pytest.skip(str(e))
    exe = tmp_path / "gfft_host"
    subprocess.run([nvcc, "-O1", "-std=c++17", "-arch=sm_103a", "-I", os.path.join(ROOT, "paper_1112_1805_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "gfft_host.cu"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert r.stdout.rstrip().endswith("bad 0")
