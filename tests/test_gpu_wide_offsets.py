"""The odd step with 64-bit offsets, which domains take from 4 GB of populations on, over every form a step has: the
runtime is compiled so that every domain takes it (the kernels are those of the library) and the parity cases of the
bounds-checked build run against that library in a child process."""
import glob
import os
import subprocess
import sys

import pytest

from paper_2502_12955_gb300 import build as lbm_build
from tests.test_gpu_bounds import CASES, ROOT

pytestmark = pytest.mark.gpu


def test_parity_cases_with_64_bit_offsets():
    lbm_build.build()
    out = os.path.join(lbm_build.BUILD, "wide_offsets")
    os.makedirs(out, exist_ok=True)
    nvcc, obj, lib = lbm_build._nvcc(), os.path.join(out, "runtime.o"), os.path.join(out, "liblbm.so")
    others = [o for o in glob.glob(os.path.join(lbm_build.BUILD, "*.o")) if os.path.basename(o) != "runtime.o"]
    for cmd in ([nvcc, *lbm_build.ARCH, *lbm_build.NVFLAGS, "-DLBM_OFF32_BYTES=0", "-c",
                 os.path.join(lbm_build.CSRC, "runtime.cu"), "-o", obj],
                [nvcc, *lbm_build.ARCH, "-shared", "-cudart", "static", "-o", lib, obj, *others]):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-2000:]
    cases = CASES + ["test_gpu_routes.py", "test_gpu_conservation.py"]
    cmd = [sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider"]
    cmd += [os.path.join(ROOT, "tests", c) for c in cases]
    r = subprocess.run(cmd, cwd=ROOT, env=dict(os.environ, LBM_LIBRARY=lib), capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, (r.stdout + r.stderr)[-3000:]
