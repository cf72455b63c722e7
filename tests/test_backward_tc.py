"""The FP64 adjoint by digit products on the tensor cores (default for ADVDIFF and most of HELMHOLTZ) against
the plain FP64 kernel (FLAG_CUDA_CORES through the C arguments); test_backward.py holds the default against the
oracle.

Tolerance against the plain kernel, of max|gradient|: both kernels' factor gradients carry at most (N + 8)
roundings of 2^-53 of sums of N products, the chain some 50 more of terms up to 2^4 times the result, and a
node adds up 24 cells: (N + 64) 2^-47. Below 2^-1022 a rounding is no longer relative but 2^-1075: (N + 64) of
those, times the 2^10 or less by which the chain multiplies them here, add (N + 64) 2^-1064.
"""
import ctypes

import numpy as np
import pytest
import torch

import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import binding as B
from paper_1407_0904_gb300 import meshgen
from tests.helpers import TRI, TET, HELMHOLTZ, ADVDIFF, FP64, coefficients, to_device

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CASES = [(HELMHOLTZ, TRI, 2), (HELMHOLTZ, TRI, 3)] + [(HELMHOLTZ, TET, k) for k in (1, 2, 3, 4)]
CASES += [(ADVDIFF, c, k) for c in (TRI, TET) for k in (1, 2, 3, 4)]


def backward(form, k, cell, args, dout, flags=0, deterministic=0, validate=False):
    x, c2v, cf, cd = args
    a, _ = B.make_args(form, k, cell, x, c2v, cf, cd, FP64, dout, 0.01, validate, tune=flags)
    dx = torch.zeros_like(x)
    dc = torch.zeros_like(cf) if cf is not None else None
    B._check(coffee.lib().coffee_assemble_backward(ctypes.byref(a), B._ptr(dout), B._ptr(dx), B._ptr(dc), deterministic,
                                                   B._stream_handle(None)))
    return [dx] + ([dc] if dc is not None else [])


def inputs(form, cell, k, ncells, seed=7):
    n = 1
    while (2 * n * n if cell == TRI else 6 * n ** 3) < ncells:
        n += 1
    mesh = (meshgen.tri_mesh if cell == TRI else meshgen.tet_mesh)(n, seed=seed)
    mesh.cell2vert, mesh.grid = np.ascontiguousarray(mesh.cell2vert[:ncells]), mesh.grid[:ncells]
    coef, c2d = coefficients(form, mesh, k, seed)
    n = coffee.ndof(form, k, cell)
    dout = np.random.default_rng(seed).standard_normal((ncells, n, n))
    return mesh, coef, c2d, dout


def close(a, b, N):
    for g, w in zip(a, b):
        assert float((g - w).abs().max()) <= (N + 64) * 2.0 ** -47 * float(w.abs().max())


@pytest.mark.parametrize("form,cell,k", CASES)
@pytest.mark.parametrize("ncells", [1, 129, 20011])  # one row of a tile, one past a tile, tiles on both sets of warps
def test_against_plain(form, cell, k, ncells):
    mesh, coef, c2d, dout = inputs(form, cell, k, ncells)
    args, d = to_device(mesh, coef, c2d, DEV), torch.from_numpy(dout).to(DEV)
    got = backward(form, k, cell, args, d, validate=True)
    coffee.check_errors()
    close(got, backward(form, k, cell, args, d, coffee.FLAG_CUDA_CORES), dout[0].size)


@pytest.mark.parametrize("form,cell,k", [(HELMHOLTZ, TET, 3), (ADVDIFF, TRI, 3)])
def test_gradients_outside_the_digits_range(form, cell, k):
    """Rows of dA that are zero, tiny, subnormal, huge, of very different size, or hold an infinity or NaN, every
    cell on vertices of its own: as the plain kernel gives them."""
    mesh, coef, c2d, dout = inputs(form, cell, k, 140)
    X = mesh.coords[mesh.cell2vert]
    mesh.coords = np.ascontiguousarray(X.reshape(-1, X.shape[2]))
    nv = X.shape[1]
    mesh.cell2vert = np.arange(140 * nv, dtype=np.int32).reshape(140, nv)
    dout[3] = 0.0
    dout[4] *= 1e-290
    dout[5] = 5e-324
    dout[6] *= 1e280
    dout[7] *= np.exp(np.random.default_rng(1).uniform(-60, 60, dout[7].shape))
    dout[60, 1, 2] = np.inf
    dout[61, 0, 0] = np.nan
    dout[62] = -0.0
    args, d = to_device(mesh, coef, c2d, DEV), torch.from_numpy(dout).to(DEV)
    a = backward(form, k, cell, args, d)[0].reshape(140, -1).cpu().numpy()
    b = backward(form, k, cell, args, d, coffee.FLAG_CUDA_CORES)[0].reshape(140, -1).cpu().numpy()
    fine = np.isfinite(b)
    assert np.array_equal(fine.all(1), np.isfinite(a).all(1))
    rows = fine.all(1)
    big = np.abs(b[rows]).max(1, keepdims=True)
    assert np.all(np.abs(a[rows] - b[rows]) <= (dout[0].size + 64) * (2.0 ** -47 * big + 2.0 ** -1064))


def test_deterministic_of_many_cells_and_bad_index():
    """Above the allocation-free entry point's limit the deterministic adjoint runs here too, the same every time;
    a cell with an index out of range contributes nothing."""
    mesh, coef, c2d, dout = inputs(ADVDIFF, TET, 1, 20000)
    args, d = to_device(mesh, coef, c2d, DEV), torch.from_numpy(dout).to(DEV)
    a, b = (backward(ADVDIFF, 1, TET, args, d, deterministic=1) for _ in range(2))
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    close(a, backward(ADVDIFF, 1, TET, args, d), 16)
    x, c2v, cf, cd = args
    bad = c2v.clone()
    bad[777, 2] = -1
    got = backward(ADVDIFF, 1, TET, (x, bad, cf, cd), d, validate=True)
    with pytest.raises(coffee.CoffeeError):
        coffee.check_errors()
    d2 = d.clone()
    d2[777] = 0.0
    close(got, backward(ADVDIFF, 1, TET, args, d2), 16)
