"""FP64 element matrices entry by entry: every entry to double rounding of its own terms, sum_k |G_k T_k|, also where
that is far below the cell's largest entry (right-angled cells, thin layers, flow along an axis), as the plain
kernel (FLAG_CUDA_CORES) gives them.

Tolerances, in units of 2^-53 of sum_k |G_k T_k|, against the plain kernel, which forms the factors by the same
operations but for the divisions (a rounding more): K roundings there. By digits an entry has a term of 2^-8 of
max|G| max|T| or more: per factor 2^-60.4 from the two truncations and 2^-58.4 from the products left out, 2^-58 of
that scale in all or 8 units; the sums' low bits 4 (b = 9, steps of 2^-59) or 64 (b = 8, 2^-56), and values below
four steps become zero: 16 or 128. Together 10 K + 28, with 8-bit digits (advection-diffusion) 10 K + 200. The root mean
square of the differences, of which few reach that, within that of K random roundings each, 2 sqrt(K).
"""
import numpy as np
import pytest
import torch

import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import meshgen
from tests.helpers import TRI, TET, HELMHOLTZ, ADVDIFF, to_device

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def mesh_of(cell, stretch, perturb):
    mesh = meshgen.tri_mesh(13, perturb=perturb) if cell == TRI else meshgen.tet_mesh(4, perturb=perturb)
    mesh.coords = mesh.coords * 0.125
    mesh.coords[:, -1] *= stretch
    return mesh


def coefficients(mesh, eps, axis):
    rng = np.random.default_rng(2)
    nn, d = mesh.coords.shape
    rows = np.concatenate([eps * (0.5 + rng.random((nn, 1))), 2 * rng.random((nn, d)) - 1], 1)
    if axis:
        rows[:, 1:] = np.eye(d)[0]
    return rows.reshape(-1), mesh.cell2vert


def factors(form, mesh, coef, c2d):
    """G [cells, K] in extended precision."""
    X = mesh.coords[mesh.cell2vert].astype(np.longdouble)
    d = X.shape[2]
    J = np.swapaxes(X[:, 1:] - X[:, :1], 1, 2)
    cols = [J[:, :, a] for a in range(d)]
    if d == 2:
        adj = np.stack([np.stack([cols[1][:, 1], -cols[1][:, 0]], 1), np.stack([-cols[0][:, 1], cols[0][:, 0]], 1)], 1)
    else:
        adj = np.stack([np.cross(cols[1], cols[2]), np.cross(cols[2], cols[0]), np.cross(cols[0], cols[1])], 1)
    det = (cols[0] * adj[:, 0]).sum(1)
    H = np.stack([(adj[:, a] * adj[:, b]).sum(1) / abs(det) for a in range(d) for b in range(a, d)], 1)
    if form == HELMHOLTZ:
        return np.concatenate([abs(det)[:, None], H], 1)
    rows = coef.reshape(-1, d + 1)[c2d].astype(np.longdouble)
    stiff = (rows[:, :, :1] * H[:, None, :]).reshape(len(H), -1)
    adv = np.einsum("nar,nvr->nva", adj * np.sign(det)[:, None, None], rows[:, :, 1:]).reshape(len(H), -1)
    return np.concatenate([stiff, adv], 1)


CASES = [(HELMHOLTZ, TRI, 2), (HELMHOLTZ, TRI, 3), (HELMHOLTZ, TET, 1), (HELMHOLTZ, TET, 2), (HELMHOLTZ, TET, 3), (HELMHOLTZ, TET, 4),
         (ADVDIFF, TRI, 2), (ADVDIFF, TRI, 4), (ADVDIFF, TET, 1), (ADVDIFF, TET, 2), (ADVDIFF, TET, 3)]


@pytest.mark.parametrize("form,cell,k", CASES)
@pytest.mark.parametrize("stretch,perturb,eps,axis", [(1, 0.0, 1.0, False), (1e-3, 0.1, 1e-6, False), (1e-3, 0.0, 1.0, True),
                                                      (1e-6, 0.0, 1e-6, True)])
def test_every_entry_to_rounding_of_its_terms(form, cell, k, stretch, perturb, eps, axis):
    mesh = mesh_of(cell, stretch, perturb)
    coef, c2d = coefficients(mesh, eps, axis) if form == ADVDIFF else (None, None)
    args = to_device(mesh, coef, c2d, DEV)
    nc = mesh.cell2vert.shape[0]
    A = coffee.assemble(form, k, cell, *args, validate=True)
    n = A.shape[1]
    M = coffee.CsrMatrix(torch.arange(nc * n, dtype=torch.int32, device=DEV).view(nc, n), nc * n)  # an entry a value
    assert torch.equal(M.assemble(form, k, cell, *args).view_as(A), A)
    coffee.check_errors()
    G = factors(form, mesh, coef, c2d)
    T = np.asarray(coffee.reference_tensor(form, k, cell)).reshape(G.shape[1], -1).astype(np.longdouble)
    plain = coffee.assemble(form, k, cell, *args, tune=coffee.FLAG_CUDA_CORES).cpu().numpy().reshape(nc, -1)
    got, size = A.cpu().numpy().reshape(nc, -1), abs(G) @ abs(T)
    err = abs(got - plain) / np.where(size > 0, size, 1) * 2.0 ** 53
    K = G.shape[1]
    assert np.all(got[size == 0] == 0)
    assert float(err.max()) <= 10 * K + (28 if form == HELMHOLTZ else 200)
    assert float(np.sqrt((err ** 2).mean())) <= 2 * K ** 0.5


@pytest.mark.parametrize("form,cell,k", [(HELMHOLTZ, TRI, 3), (HELMHOLTZ, TET, 2), (ADVDIFF, TET, 2)])
def test_global_values_of_cells_without_digits(form, cell, k):
    """Cells with a NaN coordinate, flat, tiny or huge, among ordinary ones in one tile of the fused global assembly:
    each value is the element matrix's entry."""
    mesh = mesh_of(cell, 1.0, 0.1)
    X = mesh.coords[mesh.cell2vert][:77].copy()
    X[3] *= 1e-160
    X[17] *= 1e120
    X[50, 2] = X[50, 1]
    X[51, 0, 0] = np.nan
    mesh.coords = np.ascontiguousarray(X.reshape(-1, X.shape[2]))
    mesh.cell2vert = np.arange(X.shape[0] * X.shape[1], dtype=np.int32).reshape(X.shape[:2])
    coef, c2d = coefficients(mesh, 1.0, False) if form == ADVDIFF else (None, None)
    args = to_device(mesh, coef, c2d, DEV)
    A = coffee.assemble(form, k, cell, *args)
    n = A.shape[1]
    M = coffee.CsrMatrix(torch.arange(77 * n, dtype=torch.int32, device=DEV).view(77, n), 77 * n)
    assert torch.equal(torch.nan_to_num(M.assemble(form, k, cell, *args).view_as(A), nan=7.5), torch.nan_to_num(A, nan=7.5))
    plain = coffee.assemble(form, k, cell, *args, tune=coffee.FLAG_CUDA_CORES)
    # the sums of the plain kernel: K roundings each, and some of the factors' (the determinants of 3 and 50 are rounding
    # or subnormal, so their factors have no digits in common; that of 17 overflows in 3D)
    K = np.asarray(coffee.reference_tensor(form, k, cell)).shape[0]
    fine = plain[17].isfinite()
    assert torch.equal(A[17].isfinite(), fine) and (cell == TET or bool(fine.all()))
    diff, size = (torch.where(fine, x, 0.0).abs().max() for x in (A[17] - plain[17], plain[17]))
    assert float(diff) <= (2 * K + 16) * 2.0 ** -50 * float(size)
    assert bool(A[51].isnan().all()) and bool(plain[51].isnan().all())
