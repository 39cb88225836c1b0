"""The package's lazily imported names (no GPU)."""

import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_serve_is_an_attribute_of_the_package():
    code = ("import paper_2509_19162_gb300 as p; assert p.serve.Server.__name__ == 'Server'; "
            "assert p.Growth and p.Batch; from paper_2509_19162_gb300 import serve; assert serve is p.serve")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-500:]
