"""Device memory that mesh creation reaches for: the maps (material, ranks, row
pointers, columns, element slots: 375 bytes an element of a 160^3 box), the row
masks (4) and two words of six faces (48), in a process of its own."""
import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu

ROOT = Path(__file__).resolve().parents[1]
CHILD = """
import torch
from paper_0704_2344_gb300 import fe, workloads as W
ctx = fe.fe_ctx_create(0)
prob = W.empty_box(160)
before = torch.cuda.mem_get_info()[0]
mesh = fe.fe_mesh_create_from(ctx, prob)
fe.fe_ctx_synchronize(ctx)
print((before - torch.cuda.mem_get_info()[0]) / 160 ** 3)
"""


def test_mesh_creation_peak():
    out = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    assert float(out.stdout.split()[-1]) <= 427 + 15  # allocations round up to 32 MiB (8 bytes an element) at most twice
