"""Element matrices of prisms in every tensor-core precision are made of the operand parts that the precision
names: the same as the global assembly of the same cells, whose kernel contracts all points with those parts. Every
cell has nodes of its own, so that a matrix value is one entry added to zero, and the two have the same bits; in
split tf32, where element matrices are summed direction by direction, they agree to that precision's bound."""
import numpy as np
import pytest
import torch

import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import meshgen
from tests.helpers import MASS, HELMHOLTZ, ADVDIFF, TF32, TF32X3, BF16, BF16X3, TOL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
P = coffee.PRISM


@pytest.mark.parametrize("form", [MASS, HELMHOLTZ, ADVDIFF])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
def test_local_and_global_have_the_same_operands(form, k):
    mesh = meshgen.prism_mesh(5, 6, perturb=0.15, seed=4)
    c2v, coef, c2d = mesh.cell2vert, None, None
    if form == ADVDIFF:
        coef, c2d, _ = meshgen.advdiff_coefficients(mesh, 3)
    t = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    args = [t(mesh.coords), t(c2v), t(coef), t(c2d)]
    nc, n = c2v.shape[0], coffee.ndof(form, k, P)
    M = coffee.CsrMatrix(torch.arange(nc * n, dtype=torch.int32, device=DEV).view(nc, n), nc * n)
    assert M.nnz == nc * n * n
    for prec in (TF32, TF32X3, BF16, BF16X3):
        A = coffee.assemble(form, k, P, *args, precision=prec, validate=True)
        vals = M.assemble(form, k, P, *args, precision=prec).view(nc, n, n)
        coffee.check_errors()
        if prec == TF32X3 and form != MASS:
            big = A.abs().flatten(1).amax(1)[:, None, None]
            assert float(((A - vals).abs() / big).max()) < 2 * TOL[prec]
        else:
            assert torch.equal(A, vals)
