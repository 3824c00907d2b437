"""The launch shape when the blocks' state buffer cannot be had: shared-memory
state or fewer blocks, the same results, and no buffer freed and allocated again
from call to call (tests/state_memory.cu, linked with the library's objects and
a cudaMalloc that refuses large requests)."""
import glob
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_batches_with_little_memory(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_03549_gb300 import build

    build.build_library()
    objs = sorted(glob.glob(os.path.join(build.BUILD, "*.cu.o")))
    assert len(objs) == len(build._sources())
    exe = str(tmp_path / "state_memory")
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I",
                    build.INCLUDE, "-I", build.CSRC, "-Xlinker",
                    "--wrap=cudaMalloc", "-o", exe,
                    os.path.join(HERE, "state_memory.cu"), *objs],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
