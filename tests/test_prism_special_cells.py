"""Prisms with a NaN coordinate, flat (no volume) or inverted beside ordinary ones, in tiles of the tensor-core kernels and
blocks of the FP64 one: the ordinary cells' matrices are the ones they have alone, the NaN cell's are NaN."""
import numpy as np
import pytest
import torch

import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import meshgen
from tests.helpers import HELMHOLTZ, ADVDIFF, FP64, TF32X3, BF16

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
P = coffee.PRISM


@pytest.mark.parametrize("form", [HELMHOLTZ, ADVDIFF])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("prec", [FP64, TF32X3, BF16])
def test_special_cells_beside_ordinary_ones(form, k, prec):
    mesh = meshgen.prism_mesh(4, 3, perturb=0.1, seed=5)
    X = mesh.coords[mesh.cell2vert]
    n = len(X)
    X[5, 3, 1] = np.nan
    X[30, 3:] = X[30, :3]              # flat: divisions by zero
    X[31] = X[31][[3, 4, 5, 0, 1, 2]]  # upside down: a negative determinant, which the measure accepts
    coef = c2d = None
    if form == ADVDIFF:
        c, idx, _ = meshgen.advdiff_coefficients(mesh, 3)
        coef = np.ascontiguousarray(c.reshape(-1, 4)[idx].reshape(-1))
        c2d = np.arange(6 * n, dtype=np.int32).reshape(n, 6)
    t = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    x, c2v, cf = t(X.reshape(-1, 3)), t(np.arange(6 * n, dtype=np.int32).reshape(n, 6)), t(coef)
    run = lambda rows: coffee.assemble(form, k, P, x, c2v[rows].contiguous(), cf,
                                       None if c2d is None else t(c2d)[rows].contiguous(), precision=prec)
    rows = torch.arange(n, device=DEV)
    good = rows[(rows != 5) & (rows != 30)]
    A = run(rows)
    assert bool(A[5].isnan().all()) and bool(A[good].isfinite().all())
    assert torch.equal(A[good], run(good))
