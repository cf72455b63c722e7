"""Which launches take the sector-aligned stores: both sides of every threshold of cells, strides, precisions and knobs; and,
on the GPU, rows of four offsets (strides 2 modulo 4) against the other kernel, which a knob asks for."""
import numpy as np
import pytest
import torch

import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import binding as B
from paper_1407_0904_gb300 import meshgen
from tests.helpers import TRI, TET, MASS, HELMHOLTZ, ADVDIFF, BURGERS_JAC, FP64, TF32, TF32X3, BF16, BF16X3

DEV = "cuda:0"


@pytest.mark.parametrize("form,k,cell,prec,stride,least", [
    (HELMHOLTZ, 4, TET, TF32X3, 0, 16384), (MASS, 4, TET, TF32, 0, 16384), (HELMHOLTZ, 4, TET, BF16X3, 0, 32768),
    (HELMHOLTZ, 4, TET, BF16, 1227, 16384), (HELMHOLTZ, 4, TRI, BF16, 0, 16384), (ADVDIFF, 4, TRI, TF32, 0, 16384),
    (HELMHOLTZ, 4, TRI, TF32X3, 0, 131072), (HELMHOLTZ, 3, TET, TF32X3, 402, 131072), (HELMHOLTZ, 3, TET, BF16, 402, 16384),
    (HELMHOLTZ, 3, TET, BF16, 404, 16384)])
def test_thresholds(form, k, cell, prec, stride, least):
    use = lambda n, flags=0: B.diag_sector_stores(form, k, cell, prec, flags, stride, n)
    assert use(least) and not use(least - 1)
    for knob in (coffee.FLAG_OUTPUT_LANES, coffee.FLAG_TWO_STAGES, coffee.FLAG_SUBTILE_64, coffee.FLAG_SUBTILE_32,
                 coffee.FLAG_SUBTILE_128, coffee.FLAG_CELL_LANES, coffee.FLAG_STAGED_STORE):
        assert not use(least, knob) and use(least, knob | B.FLAG_KNOB_HINT)
    assert use(least, B._tuned_flags(form, k, cell, prec))  # the autotuner's knobs do not keep a launch from it


@pytest.mark.parametrize("form,k,cell,prec,stride", [
    (HELMHOLTZ, 3, TET, TF32X3, 0), (HELMHOLTZ, 3, TET, BF16, 408), (HELMHOLTZ, 3, TET, BF16X3, 402), (ADVDIFF, 4, TRI, TF32X3, 0),
    (HELMHOLTZ, 2, TET, TF32, 101), (BURGERS_JAC, 2, TET, TF32X3, 0), (HELMHOLTZ, 4, coffee.PRISM, TF32X3, 0), (HELMHOLTZ, 4, TET, FP64, 0)])
def test_never(form, k, cell, prec, stride):
    assert not B.diag_sector_stores(form, k, cell, prec, 0, stride, 1 << 24)


def test_arguments_out_of_range():
    with pytest.raises(coffee.CoffeeError):
        B.diag_sector_stores(HELMHOLTZ, 5, TET, TF32X3)


@pytest.mark.gpu
@pytest.mark.parametrize("stride,shift", [(402, 0), (402, 3), (406, 1)])
def test_rows_of_four_offsets(stride, shift):
    ncells = 17003
    assert B.diag_sector_stores(HELMHOLTZ, 3, TET, BF16, 0, stride, ncells)
    mesh = meshgen.tet_mesh(15, seed=8, ncells=ncells)
    x, c2v = torch.from_numpy(mesh.coords).to(DEV), torch.from_numpy(np.ascontiguousarray(mesh.cell2vert)).to(DEV)
    flat = torch.full((8 + ncells * stride,), 9.0, device=DEV)
    out = flat[shift:shift + ncells * stride]
    coffee.assemble(HELMHOLTZ, 3, TET, x, c2v, precision=BF16, out=out, out_stride=stride, validate=True, tune=0)
    want = coffee.assemble(HELMHOLTZ, 3, TET, x, c2v, precision=BF16, tune=coffee.FLAG_SUBTILE_128)
    coffee.check_errors()
    rows = out.view(ncells, stride)
    assert torch.equal(rows[:, :400], want.view(ncells, 400)) and bool((rows[:, 400:] == 9.0).all())
    assert bool((flat[:shift] == 9.0).all()) and bool((flat[shift + ncells * stride:] == 9.0).all())
