"""The autotuner's file: lines of the present version are used, older ones (chosen
against other default kernels) are passed over and their case is timed again."""

import os
import subprocess
import sys

import pytest

TUNE = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
import gen
from gpu_util import to_device
import paper_2303_08609_gb300 as weo
op = weo.WilsonEO((8, 8, 8, 8), 0.13, to_device(gen.gauge_field((8, 8, 8, 8), "haar", seed=1201)), prec="f32")
print("ms", weo.wilson_eo_tune(op.handle)[2])
"""


def tune(path):
    tests = os.path.dirname(os.path.abspath(__file__))
    code = TUNE.format(root=os.path.dirname(tests), tests=tests)
    r = subprocess.run([sys.executable, "-c", code], env={**os.environ, "WILSON_EO_TUNE_CACHE": str(path)},
                       capture_output=True, text=True, check=True)
    return float(r.stdout.split()[-1])


@pytest.mark.gpu
def test_lines_of_this_and_of_older_versions(tmp_path):
    path = tmp_path / "tune.txt"
    ms = tune(path)
    (line,) = path.read_text().splitlines()
    version, key, *fields = line.split()
    assert 0 < ms < 100 and version == "v8" and len(fields) == 10
    fields[5] = "123.0"
    path.write_text(" ".join([version, key, *fields]) + "\n")
    assert tune(path) == 123.0 and len(path.read_text().splitlines()) == 1
    for n, old in ((10, "v7"), (9, "v6"), (6, "v3")):
        path.write_text(" ".join([old, key, *fields[:n]]) + "\n")
        assert tune(path) < 100
        lines = path.read_text().splitlines()
        assert len(lines) == 2 and lines[1].startswith("v8 " + key)
