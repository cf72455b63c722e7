"""Sector-aligned stores of element matrices that start off the 32-byte sectors (P4, or odd padded rows), which the
library takes from 16384 cells on: the same bits as the same cells assembled in launches too small for it, and
the oracle's matrices within each precision's bound."""
import numpy as np
import pytest
import torch

import paper_1407_0904_gb300 as coffee
from tests.helpers import (TRI, TET, MASS, HELMHOLTZ, ADVDIFF, TF32, TF32X3, BF16, BF16X3, TOL, coefficients, oracle_ref,
                           rel_err_per_cell, small_mesh, to_device)

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def problem(form, cell, k, ncells):
    mesh = small_mesh(cell, n=int(np.ceil((ncells / (2 if cell == TRI else 6)) ** (0.5 if cell == TRI else 1 / 3))), seed=8)
    mesh.cell2vert, mesh.grid = np.ascontiguousarray(mesh.cell2vert[:ncells]), mesh.grid[:ncells]
    coef, c2d = coefficients(form, mesh, k)
    return mesh, coef, c2d


@pytest.mark.parametrize("form,cell,k,prec,ncells,stride,shift", [
    (HELMHOLTZ, TET, 4, TF32X3, 16385, 0, 0), (MASS, TET, 4, TF32, 20011, 0, 3), (HELMHOLTZ, TET, 4, BF16X3, 33001, 0, 5),
    (HELMHOLTZ, TRI, 4, BF16, 40003, 0, 1), (ADVDIFF, TRI, 4, TF32, 38911, 0, 0), (HELMHOLTZ, TRI, 4, TF32X3, 131072, 0, 0),
    (HELMHOLTZ, TET, 3, TF32X3, 17000, 402, 0), (HELMHOLTZ, TET, 3, BF16, 16999, 404, 2), (HELMHOLTZ, TET, 4, BF16, 16384, 1227, 7)])
def test_same_bits_as_small_launches(form, cell, k, prec, ncells, stride, shift):
    """stride: padded rows of 2, 4 or 8 offsets; shift: floats by which the output starts off a sector."""
    mesh, coef, c2d = problem(form, cell, k, ncells)
    x, c2v, cf, cd = to_device(mesh, coef, c2d, DEV)
    n2 = coffee.ndof(form, k, cell) ** 2
    row = stride or n2
    flat = torch.full((8 + ncells * row,), 9.0, device=DEV)
    out = flat[shift:shift + ncells * row]
    coffee.assemble(form, k, cell, x, c2v, cf, cd, precision=prec, out=out, out_stride=stride or None, validate=True)
    coffee.check_errors()
    got = out.view(ncells, row)[:, :n2]
    for lo in range(0, ncells, 16000):
        hi = min(lo + 16000, ncells)
        want = coffee.assemble(form, k, cell, x, c2v[lo:hi].contiguous(), cf, None if cd is None else cd[lo:hi].contiguous(),
                               precision=prec)
        assert torch.equal(got[lo:hi], want.view(hi - lo, n2))
    assert bool((out.view(ncells, row)[:, n2:] == 9.0).all())
    assert bool((flat[:shift] == 9.0).all()) and bool((flat[shift + ncells * row:] == 9.0).all())
    sel = np.array([0, ncells // 3, ncells - 1])
    ref = oracle_ref(form, k, cell, mesh, coef, c2d, sel).reshape(3, -1)
    assert rel_err_per_cell(got[torch.from_numpy(sel).to(DEV)].cpu().numpy(), ref) < TOL[prec]
