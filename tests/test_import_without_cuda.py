"""The package imports, and problems and settings can be made, with a PyTorch
that was built without CUDA (whose torch._C has no _cuda_ functions)."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import torch
for name in [n for n in dir(torch._C) if n.startswith("_cuda_")]:
    delattr(torch._C, name)
from paper_1208_0302_gb300 import api
pb = api.Problem([(6302.5017, 2.5, 1.0)], [6302.0 + 0.01 * i for i in range(64)], 6302.5017)
assert pb.n_lambda == 64 and api.bounds(range(9), range(1, 10)).hi[8] == 9.0
assert api.GaSettings().to_c(0).npop == 128
try:
    api.me_synth(pb, torch.zeros((1, 9), dtype=torch.float64))
except ValueError as e:
    assert "CUDA tensor" in str(e)
else:
    raise SystemExit("a CPU tensor was accepted")
"""


def test_import_without_cuda():
    done = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True)
    assert done.returncode == 0, done.stderr
