"""The package imports where torch was built without CUDA (its host parts, the layout
and synthetic helpers, need none)."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_import_without_cuda_in_torch():
    code = ("import torch; vars(torch._C).pop('_cuda_getCurrentRawStream', None); "
            "from paper_1202_6522_gb300 import SHT, UnevenBatch, synthetic; synthetic.spectrum(3)")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
