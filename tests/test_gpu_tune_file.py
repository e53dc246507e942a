"""Saved product choices: used when they were made among the kernels of this
library, passed over when the file is from before them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import torch
import ed_inputs as ei
from paper_2308_16712_gb300 import ed
h = ei.heisenberg_ring(20)
O = ed.operator_create(20, h["sites"], h["coeff"], h["local"])
B = ed.basis_build(20, 10, +1, *ei.ring_group(20, 0, +1))
x = torch.rand(ed.basis_size(B), dtype=torch.float64, device="cuda")
if {tune}:
    ed.autotune(O, B, x, torch.empty_like(x))
before = ed.product_counts()
ed.matvec(O, B, x, torch.empty_like(x))
torch.cuda.synchronize()
print([k for k, v in ed.product_counts().items() if v > before[k]][0])
"""


def run(path, tune=False):
    out = subprocess.run([sys.executable, "-c", PROGRAM.format(tune=tune)], cwd=ROOT, check=True, timeout=300,
                         env=dict(os.environ, ED_TUNE_FILE=str(path)), capture_output=True, text=True)
    return out.stdout.split("\n")[0]


def test_saved_choices(tmp_path):
    path = tmp_path / "tune.txt"
    run(path, tune=True)
    fields = path.read_text().split("\n")[0].split()
    assert fields[0] == "P" and len(fields) == 12
    current, older = fields[:], fields[:-1]
    for line in (current, older):
        line[9:11] = ["1", "0"]  # row-per-lane, every rotation
    path.write_text("\n".join([" ".join(current), ""]))
    assert run(path) == "row-per-lane"
    path.write_text("\n".join([" ".join(older), ""]))
    assert run(path) == "slot without copy"  # a small sector
    path.write_text("\n".join([" ".join(older), " ".join(current), ""]))
    assert run(path) == "row-per-lane"
