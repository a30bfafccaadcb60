"""The file of measured kernel times: what this library measured is read back by a later process, times
of another generation of the kernels are not."""
import os
import subprocess
import sys

import pytest

from paper_2604_17109_gb300 import build as pkg_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

REPORT = "from paper_2604_17109_gb300 import pim; print(pim.pim_tune_report())"
MEASURE = """
import numpy as np
from paper_2604_17109_gb300 import pim
hd = pim.pim_create(np.triu(np.ones((300, 300), np.int8), 1) + np.tril(np.ones((300, 300), np.int8), -1), None, 0.1)
pim.pim_set_schedule(hd, np.linspace(0.1, 3, 40), np.ones(40), 0.5)
pim.pim_batch_destroy(pim.pim_batch_create([hd], [64]))
print(pim.pim_tune_report())
"""


def _python(script, path):
    pkg_build.build()
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, PIM_TUNE_CACHE=str(path)))
    assert r.returncode == 0, r.stderr
    return r.stdout.strip().splitlines()


def test_times_of_older_kernels_are_passed_over(tmp_path):
    path = tmp_path / "times"
    path.write_text("NVIDIA_GB300|mid|512|256|0|0 8.3\nkernels1 NVIDIA_GB300|fused|128|1|0|0 4.5\nnoise\n")
    assert _python(REPORT, path) == []


@pytest.mark.gpu
def test_measured_times_are_read_back(tmp_path):
    path = tmp_path / "times"
    path.write_text("NVIDIA_GB300|mid|512|256|0|0 8.3\n")
    first = _python(MEASURE, path)
    assert any("|mid|" in line for line in first) and any("|big|" in line for line in first)
    again = _python(REPORT, path)
    assert [line.split()[0] for line in again] == [line.split()[0] for line in first]
    for a, b in zip(again, first):
        assert float(a.split()[1]) == pytest.approx(float(b.split()[1]), rel=2e-3)  # four digits each
    assert len(path.read_text().splitlines()) == 1 + len(first)
