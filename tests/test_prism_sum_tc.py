"""Prisms on the tensor cores with the quadrature summed over z first (HELMHOLTZ, ADVDIFF): cell counts around the
tiles of CELLS cells (a quarter of one per TMEM lane quadrant), blocks with several tiles, outputs off the vector
alignment, invalid cells. Every precision runs the split-tf32 operands, so the split precisions' bound
(tests.helpers.TOL) holds for all four, against the oracle's sum over the same rule."""
import numpy as np
import pytest
import torch

import oracle
import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import meshgen
from tests.helpers import HELMHOLTZ, ADVDIFF, TF32, TF32X3, BF16, BF16X3, TOL, rel_err_per_cell

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
P = coffee.PRISM
CELLS = {HELMHOLTZ: (40, 20, 12, 8), ADVDIFF: (32, 12, 8, 4)}


def problem(form, n, nz, ncells):
    mesh = meshgen.prism_mesh(n, nz, perturb=0.15, seed=12)
    assert mesh.cell2vert.shape[0] >= ncells
    c2v, coef, c2d = np.ascontiguousarray(mesh.cell2vert[:ncells]), None, None
    if form == ADVDIFF:
        coef, c2d, _ = meshgen.advdiff_coefficients(mesh, 3)
        c2d = np.ascontiguousarray(c2d[:ncells])
    t = lambda a: None if a is None else torch.from_numpy(a).to(DEV)
    ref = lambda k, sel: oracle.prism_assemble(form, k, mesh.coords, c2v[sel], coef, None if c2d is None else c2d[sel])
    return [t(mesh.coords), t(c2v), t(coef), t(c2d)], ref


@pytest.mark.parametrize("form", [HELMHOLTZ, ADVDIFF])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("over", [-1, 0, 1])
def test_around_a_tile(form, k, over):
    ncells = CELLS[form][k - 1] + over
    args, ref = problem(form, 3, 3, ncells)
    flat = torch.full((ncells * coffee.ndof(form, k, P) ** 2 + 2,), 9.0, device=DEV)
    out = coffee.assemble(form, k, P, *args, precision=TF32X3, out=flat[1:-1], validate=True)  # off 8 and 16 bytes
    coffee.check_errors()
    assert flat[0] == 9.0 and flat[-1] == 9.0
    want = ref(k, np.arange(ncells))
    assert rel_err_per_cell(out.view(want.shape).cpu().numpy(), want) < TOL[TF32X3]
    for prec in (TF32, BF16, BF16X3):  # one operand split serves all, and the aligned stores write the same
        assert torch.equal(coffee.assemble(form, k, P, *args, precision=prec).flatten(), out.flatten())


@pytest.mark.parametrize("form,k,n,nz", [(HELMHOLTZ, 1, 48, 16), (HELMHOLTZ, 3, 32, 8), (ADVDIFF, 2, 32, 8), (ADVDIFF, 4, 16, 9)])
def test_many_tiles_a_block(form, k, n, nz):
    ncells = 2 * n * n * nz - 3
    args, ref = problem(form, n, nz, ncells)
    assert ncells > 3 * 152 * CELLS[form][k - 1]
    out = coffee.assemble(form, k, P, *args, precision=TF32X3, validate=True)
    coffee.check_errors()
    sel = np.random.default_rng(1).choice(ncells, 64, replace=False)
    sel[:2] = 0, ncells - 1
    assert rel_err_per_cell(out[torch.from_numpy(sel).to(DEV)].cpu().numpy(), ref(k, sel)) < TOL[TF32X3]


@pytest.mark.parametrize("form", [HELMHOLTZ, ADVDIFF])
def test_invalid_cell_in_a_tile(form):
    args, _ = problem(form, 3, 3, 27)
    want = coffee.assemble(form, 2, P, *args, precision=TF32X3)
    args[1][13, 2] = args[0].shape[0]
    out = torch.full_like(want, 7.0)
    coffee.assemble(form, 2, P, *args, precision=TF32X3, out=out, validate=True)
    with pytest.raises(coffee.CoffeeError):
        coffee.check_errors()
    keep = torch.arange(27) != 13
    assert torch.equal(out[keep.to(DEV)], want[keep.to(DEV)]) and bool((out[13] == 0).all())
