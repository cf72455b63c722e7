"""The FP64 prism kernel's blocks of several cells (P1: seven, residual P2: two): cell counts around them, and
an invalid cell beside valid ones in its block. Bound as in test_prism*.py: 1e-12 of each cell's largest entry
against the oracle's sum over the same rule."""
import numpy as np
import pytest
import torch

import oracle
import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import meshgen
from tests.helpers import rel_err_per_cell

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
P = coffee.PRISM
FORMS = (coffee.MASS, coffee.HELMHOLTZ, coffee.ADVDIFF, coffee.BURGERS_JAC, coffee.BURGERS_RESIDUAL)


def problem(form, k, ncells):
    mesh = meshgen.prism_mesh(2, 4, seed=9)
    c2v, coef, c2d = np.ascontiguousarray(mesh.cell2vert[:ncells]), None, None
    if form == coffee.ADVDIFF:
        coef, c2d, _ = meshgen.advdiff_coefficients(mesh, 3)
    elif form >= coffee.BURGERS_JAC:
        coef, c2d, _ = meshgen.burgers_coefficients(mesh, k, 3)
        coef = coef.ravel()
    c2d = None if c2d is None else np.ascontiguousarray(c2d[:ncells])
    if form >= coffee.BURGERS_JAC:
        ref = oracle.prism_burgers(k, mesh.coords, c2v, coef.reshape(-1, 3), c2d, residual=form == coffee.BURGERS_RESIDUAL)
    else:
        ref = oracle.prism_assemble(form, k, mesh.coords, c2v, coef, c2d)
    t = lambda a: None if a is None else torch.from_numpy(a).to(DEV)
    return [t(mesh.coords), t(c2v), t(coef), t(c2d)], ref


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("k,ncells", [(1, 1), (1, 6), (1, 7), (1, 15), (2, 1), (2, 5)])
def test_ragged_blocks(form, k, ncells):
    args, ref = problem(form, k, ncells)
    out = coffee.assemble(form, k, P, *args, validate=True)
    coffee.check_errors()
    assert rel_err_per_cell(out.cpu().numpy(), ref) < 1e-12


@pytest.mark.parametrize("form", FORMS)
def test_invalid_cell_in_a_block(form):
    args, ref = problem(form, 1, 15)
    bad = args[1].clone()
    bad[9, 4] = args[0].shape[0]
    out = torch.full(ref.shape, 7.0, dtype=torch.float64, device=DEV)
    coffee.assemble(form, 1, P, args[0], bad, *args[2:], out=out, validate=True)
    with pytest.raises(coffee.CoffeeError):
        coffee.check_errors()
    got = out.cpu().numpy()
    assert np.all(got[9] == 7.0)
    rest = np.arange(15) != 9
    assert rel_err_per_cell(got[rest], ref[rest]) < 1e-12
