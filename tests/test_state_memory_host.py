"""Host-side check of the states' memory (shf_capi.cu) when it runs out, and of what
a failed launch leaves behind.

Links the library's objects with a stand-in for the CUDA runtime
(tests/fake_cudart.cpp) that runs nothing and can make any allocation or kernel
fail, and runs tests/state_memory_host.cpp.  No GPU is needed.
"""

import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_state_memory_host(tmp_path):
    from paper_1112_1805_gb300 import build

    try:
        nvcc = os.path.realpath(build.nvcc_path())
    except RuntimeError as e:  # pragma: no cover - toolkit missing
        pytest.skip(str(e))
    objs = [os.path.join(build.PKG, "_build", s.replace(".cu", ".o")) for s in build.SOURCES]
    build.build(force=not all(os.path.exists(o) for o in objs))
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    exe = str(tmp_path / "state_memory_host")
    subprocess.run(["g++", "-std=c++17", "-O1", "-no-pie", "-I", cuda, "-I", build.INCLUDE, "-o", exe,
                    *(os.path.join(HERE, f) for f in ("state_memory_host.cpp", "fake_cudart.cpp")), *objs],
                   check=True, capture_output=True, text=True, timeout=300)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0 and "all ok" in r.stdout, r.stdout + r.stderr
