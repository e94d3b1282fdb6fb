"""A workspace's size is a function of the parameters alone.  Asking for it must not
look at a device: a size that followed the device current at the first call would not
fit another one, and a program that plans before it forks must not have started CUDA."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PLAN = """
import sys
sys.path.insert(0, sys.argv[1])
from paper_2012_04838_gb300 import binding as B
for N in B.supported_sizes():
    for prec in (B.FP32_MIXED, B.FP64):
        for dealias in (B.DEALIAS_TWO_THIRDS, B.DEALIAS_PHASE_SHIFT):
            assert B.workspace_size(B.Params(N=N, precision=prec, dealias=dealias)) > 0
"""


def test_planning_does_not_load_the_driver(tmp_path):
    from paper_2012_04838_gb300 import binding, build
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        pytest.skip("no C compiler for the stand-in driver library")
    if not os.path.exists(binding.lib_path()):
        build.build()
    # a stand-in for the driver library that leaves a mark when the runtime loads it
    mark = tmp_path / "loaded"
    src = tmp_path / "cuda.c"
    src.write_text('#include <stdio.h>\n__attribute__((constructor)) static void f(void) {'
                   ' FILE* o = fopen("%s", "w"); if (o) fclose(o); }\n' % mark)
    subprocess.check_call([cc, "-shared", "-fPIC", str(src), "-o", str(tmp_path / "libcuda.so.1")])
    env = dict(os.environ, LD_LIBRARY_PATH=str(tmp_path) + ":" + os.environ.get("LD_LIBRARY_PATH", ""))
    subprocess.check_call([sys.executable, "-c", PLAN, ROOT], env=env)
    assert not mark.exists()
