"""FP64 prisms: entries without a term of the flow are to rounding of the diffusion's terms alone. Flow along x over layers of
right-angled prisms: the basis functions of the vertices opposite to the edges along x (and above each other) do not
vary along x, so their columns have no advection, and with eps = 1e-8 what is left there is 1e-8 of the matrix.

Tolerance: both matrices are sums of at most 6^3 points of 11 terms, roundings of 2^-53 each: 2^-41 = 4.5e-13 of the largest
such entry, of which far fewer meet; against the matrix without flow 1e-12."""
import numpy as np
import pytest
import torch

import oracle
import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import meshgen
from tests.helpers import ADVDIFF, rel_err_per_cell

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
P = coffee.PRISM


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("stretch", [1.0, 1e-2])
def test_entries_without_advection(k, stretch):
    mesh = meshgen.prism_mesh(4, 2, perturb=0.0)
    coords, c2v = mesh.coords * [1.0, 1.0, stretch], np.ascontiguousarray(mesh.cell2vert[::2])  # [0, ex, ex + ey]
    rows = np.zeros((coords.shape[0], 4))
    rows[:, 0] = 1e-8
    out = []
    for b in (0.0, 1.0):
        rows[:, 1] = b
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
        A = coffee.assemble(ADVDIFF, k, P, t(coords), t(c2v), t(rows.reshape(-1)), t(c2v), validate=True)
        coffee.check_errors()
        out.append(A.cpu().numpy())
        assert rel_err_per_cell(out[-1], oracle.prism_assemble(ADVDIFF, k, coords, c2v, rows.reshape(-1), c2v)) < 1e-12
    nt = (k + 1) * (k + 2) // 2
    cols = np.arange(nt - 1, nt * (k + 1), nt)  # the vertex opposite to the edge along x, on every level
    still, flow = (A[:, :, cols] for A in out)
    assert abs(out[1]).max() > 1e3 * abs(still).max()  # (the flow's entries are far larger)
    assert abs(flow - still).max() <= 1e-12 * abs(still).max()
