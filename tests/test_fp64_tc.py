"""FP64 assembly by exact digit products on the tensor cores (the default for MASS on 10 or more nodes and
for HELMHOLTZ and ADVDIFF on 4 or more) against the oracle and against the plain FP64 kernel, which
FLAG_CUDA_CORES forces.

Tolerances. The digits leave 2^-55 of max|G| max|T| or less per factor and one rounding to double; the
plain kernel rounds K sums. Both are far within the FP64 bound of 1e-12 of max|A_e|; against each other:
(K + 2) roundings of 2^-53 of sum_k |G_k T_k|, which is below 2^5 max|A_e| on these meshes.
"""
import numpy as np
import pytest
import torch

import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import meshgen
from tests.helpers import (TRI, TET, MASS, HELMHOLTZ, ADVDIFF, FP64, TOL, coefficients, oracle_ref, rel_err_per_cell,
                           to_device)

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CASES = [(f, c, k) for f in (MASS, HELMHOLTZ, ADVDIFF) for c in (TRI, TET) for k in (1, 2, 3, 4)]


def factors(form, cell):
    d = 2 if cell == TRI else 3
    P = d * (d + 1) // 2
    return {MASS: 1, HELMHOLTZ: 1 + P, ADVDIFF: (d + 1) * (P + d)}[form]


def inputs(form, cell, k, ncells, seed=5):
    n = 1
    while (2 * n * n if cell == TRI else 6 * n ** 3) < ncells:
        n += 1
    mesh = (meshgen.tri_mesh if cell == TRI else meshgen.tet_mesh)(n, seed=seed)
    mesh.cell2vert, mesh.grid = np.ascontiguousarray(mesh.cell2vert[:ncells]), mesh.grid[:ncells]
    coef, c2d = coefficients(form, mesh, k, seed)
    return mesh, coef, c2d


@pytest.mark.parametrize("form,cell,k", CASES)
@pytest.mark.parametrize("ncells", [1, 33, 20011])  # a ragged tile of 32, one cell past it, many tiles per block
def test_against_oracle_and_plain(form, cell, k, ncells):
    mesh, coef, c2d = inputs(form, cell, k, ncells)
    args = to_device(mesh, coef, c2d, DEV)
    a = coffee.assemble(form, k, cell, *args, validate=True)
    b = coffee.assemble(form, k, cell, *args, tune=coffee.FLAG_CUDA_CORES)
    coffee.check_errors()
    sel = np.unique(np.r_[0, ncells // 2, ncells - 1])
    assert rel_err_per_cell(a.cpu().numpy()[sel], oracle_ref(form, k, cell, mesh, coef, c2d, sel)) < TOL[FP64]
    scale = b.abs().flatten(1).amax(1)
    assert float(((a - b).abs().flatten(1).amax(1) / scale).max()) <= (factors(form, cell) + 2) * 2.0 ** -48


@pytest.mark.parametrize("form,cell,k", [(MASS, TET, 2), (HELMHOLTZ, TRI, 2), (HELMHOLTZ, TET, 3), (ADVDIFF, TET, 2)])
def test_cells_outside_the_digits_range(form, cell, k):
    """Cells whose factors are tiny, huge, not finite or zero (a flat cell, a NaN coordinate) among ordinary
    ones: as the plain kernel gives them, infinities and NaN in the same places."""
    mesh, coef, c2d = inputs(form, cell, k, 96)
    X = mesh.coords[mesh.cell2vert].copy()  # every cell gets its own vertices
    for e, s in ((3, 1e-160), (17, 1e120), (40, 1e-30), (41, 1e25)):
        X[e] *= s
    X[50, 2] = X[50, 1]
    X[51, 0, 0] = np.nan
    X[70, :, 0] *= 1e-9  # a sliver: factors of very different size
    mesh.coords = np.ascontiguousarray(X.reshape(-1, X.shape[2]))
    mesh.cell2vert = np.arange(X.shape[0] * X.shape[1], dtype=np.int32).reshape(X.shape[:2])
    args = to_device(mesh, coef, c2d, DEV)
    a = coffee.assemble(form, k, cell, *args).cpu().numpy().reshape(96, -1)
    b = coffee.assemble(form, k, cell, *args, tune=coffee.FLAG_CUDA_CORES).cpu().numpy().reshape(96, -1)
    fine = np.isfinite(b)
    assert np.array_equal(fine, np.isfinite(a)) and np.array_equal(np.isnan(a), np.isnan(b))
    assert np.array_equal(np.isposinf(a), np.isposinf(b))
    big = np.where(fine, np.abs(b), 0).max(1, keepdims=True)
    big[big == 0] = 1.0
    with np.errstate(invalid="ignore", over="ignore"):
        err = np.where(fine, np.abs(a - b) / big, 0)
    assert err.max() <= (factors(form, cell) + 2) * 2.0 ** -48


@pytest.mark.parametrize("form,cell,k", [(HELMHOLTZ, TET, 3), (ADVDIFF, TRI, 4)])
def test_padded_rows_and_bad_index(form, cell, k):
    """Padding and the rows of cells with an index out of range stay as they were."""
    mesh, coef, c2d = inputs(form, cell, k, 70)
    x, c2v, cf, cd = to_device(mesh, coef, c2d, DEV)
    n = coffee.ndof(form, k, cell)
    good = coffee.assemble(form, k, cell, x, c2v, cf, cd)
    bad = c2v.clone()
    bad[37, 1] = mesh.coords.shape[0]
    out = torch.full((70, n * n + 7), 3.0, dtype=torch.float64, device=DEV)
    got = coffee.assemble(form, k, cell, x, bad, cf, cd, out=out, out_stride=n * n + 7, validate=True)
    with pytest.raises(coffee.CoffeeError):
        coffee.check_errors()
    rest = torch.arange(70, device=DEV) != 37
    assert torch.equal(got[rest], good[rest])
    assert bool((out[37] == 3.0).all()) and bool((out[:, n * n:] == 3.0).all())


@pytest.mark.parametrize("form,cell,k", [(MASS, TET, 3), (HELMHOLTZ, TET, 1), (HELMHOLTZ, TRI, 4), (ADVDIFF, TET, 2)])
def test_global_values(form, cell, k):
    """Fused into CSR: the element matrices scattered (atomics: the order of a few additions differs)."""
    mesh, coef, c2d = inputs(form, cell, k, 1001)
    args = to_device(mesh, coef, c2d, DEV)
    l2g, nn = meshgen.cell2dof(mesh, k)
    M = coffee.CsrMatrix(torch.from_numpy(l2g).to(DEV), nn)
    vals = M.assemble(form, k, cell, *args)
    A = coffee.assemble(form, k, cell, *args).cpu().numpy().reshape(1001, -1)
    coffee.check_errors()
    n = l2g.shape[1]
    pos = coffee.csr_map_unblock(M.map, 1001, n).astype(np.int64)
    want = np.zeros(M.nnz)
    np.add.at(want, pos.ravel(), A.ravel())
    size = np.zeros(M.nnz)
    np.add.at(size, pos.ravel(), np.abs(A).ravel())
    assert np.all(np.abs(vals.cpu().numpy() - want) <= 2.0 ** -46 * size + 1e-300)
