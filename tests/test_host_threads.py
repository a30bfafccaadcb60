"""Host work that is shared out among threads still ends, with the same answer, where the process can
start no thread: no exception leaves the C entry."""
import os
import subprocess
import sys

import pytest

from paper_2604_17109_gb300 import build as pkg_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import resource, sys
import numpy as np
from paper_2604_17109_gb300 import pim
n = 2100  # past the size from which the checks are shared out
J = np.zeros((n, n), dtype=sys.argv[1])
J[3, 2050] = 1  # J[2050][3] is 0
pim.lib()
size = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (size + (24 << 20), -1))  # room for the call's arrays, not for stacks
try:
    pim.pim_create(J)
except pim.PimError as e:
    print(e.code == pim.PIM_ERR_INVALID, "(3, 2050)" in str(e))
"""


@pytest.mark.parametrize("dtype", ["int8", "float32"])
def test_create_without_threads(dtype):
    pkg_build.build()
    r = subprocess.run([sys.executable, "-c", SCRIPT, dtype], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, OPENBLAS_NUM_THREADS="1"))
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["True", "True"]
