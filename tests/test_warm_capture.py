"""One call of a form, degree, cell and precision, however small, builds every table that a later call of any size, kind or
direction reads: such a call can be captured in a CUDA graph. Each case runs in a process of its own, whose tables are cold."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROLOGUE = """
import numpy as np, torch
import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import meshgen
from tests.helpers import *
DEV = "cuda:0"
t = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(DEV)

def args(mesh, n, coef=None, c2d=None):
    return [t(mesh.coords), t(mesh.cell2vert[:n]), t(coef), None if c2d is None else t(c2d[:n])]

def captured(call):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = call()
    g.replay()
    torch.cuda.synchronize()
    coffee.check_errors()
    return out
"""

CASES = {
    "sector-aligned stores": """
mesh = meshgen.tet_mesh(18)
out = torch.empty(34000, 35, 35, device=DEV)
small, large = args(mesh, 100), args(mesh, 34000)
want = coffee.assemble(HELMHOLTZ, 4, TET, *small, precision=TF32X3)
captured(lambda: coffee.assemble(HELMHOLTZ, 4, TET, *large, precision=TF32X3, out=out))
assert torch.equal(out[:100], want)
""",
    "FP64 adjoint": """
mesh = meshgen.tet_mesh(6)
coef, c2d, _ = meshgen.advdiff_coefficients(mesh, 3)
a = args(mesh, 1296, coef, c2d)
coffee.assemble(ADVDIFF, 2, TET, *a)
dout = torch.randn(1296, 10, 10, device=DEV, dtype=torch.float64)
dx, dc = torch.zeros_like(a[0]), torch.zeros_like(a[2])
captured(lambda: coffee.assemble_backward(ADVDIFF, 2, TET, a[0], a[1], dout, a[2], a[3], d_coords=dx, d_coef=dc))
assert float(dx.abs().max()) > 0 and float(dc.abs().max()) > 0
""",
    "FP64 forward after the adjoint": """
mesh = meshgen.tet_mesh(4)
a = args(mesh, 384)
coffee.assemble_backward(HELMHOLTZ, 3, TET, a[0], a[1], torch.ones(384, 20, 20, device=DEV, dtype=torch.float64), deterministic=True)
out = torch.zeros(384, 20, 20, device=DEV, dtype=torch.float64)
captured(lambda: coffee.assemble(HELMHOLTZ, 3, TET, *a, out=out))
assert float(out.abs().max()) > 0
""",
    "global assembly on prisms": """
mesh = meshgen.prism_mesh(3, 3)
a = args(mesh, 54)
l2g, nn = meshgen.cell2dof(mesh, 2)
M = coffee.CsrMatrix(t(l2g), nn)
coffee.assemble(HELMHOLTZ, 2, coffee.PRISM, *a, precision=TF32X3)
vals = torch.zeros(M.nnz, device=DEV)
captured(lambda: M.assemble(HELMHOLTZ, 2, coffee.PRISM, *a, precision=TF32X3, vals=vals))
assert float(vals.abs().max()) > 0
""",
}


@pytest.mark.parametrize("name", list(CASES))
def test_capture_after_one_small_call(name):
    r = subprocess.run([sys.executable, "-c", PROLOGUE + CASES[name]], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-2000:]
