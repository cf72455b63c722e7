"""The plain FP64 adjoint from Python: tune=FLAG_CUDA_CORES of assemble_backward and AssembleFn gives the bits of the C call with
that flag (deterministic mode, above the cells that always take the plain kernel)."""
import pytest
import torch

import paper_1407_0904_gb300 as coffee
from tests.helpers import TET, ADVDIFF, to_device
from tests.test_backward_tc import DEV, backward, inputs

pytestmark = pytest.mark.gpu


def test_plain_adjoint_is_reached():
    mesh, coef, c2d, dout = inputs(ADVDIFF, TET, 1, 20000)
    args, d = to_device(mesh, coef, c2d, DEV), torch.from_numpy(dout).to(DEV)
    want = backward(ADVDIFF, 1, TET, args, d, coffee.FLAG_CUDA_CORES, deterministic=1)
    assert not torch.equal(want[1], backward(ADVDIFF, 1, TET, args, d, deterministic=1)[1])  # two kernels
    x, c2v, cf, cd = args
    got = coffee.assemble_backward(ADVDIFF, 1, TET, x, c2v, d, cf, cd, deterministic=True, tune=coffee.FLAG_CUDA_CORES)
    assert all(torch.equal(g, w) for g, w in zip(got, want))
    x, cf = x.clone().requires_grad_(), cf.clone().requires_grad_()
    out = coffee.AssembleFn.apply(x, cf, c2v, cd, ADVDIFF, 1, TET, coffee.FP64, True, coffee.FLAG_CUDA_CORES)
    assert torch.equal(out, coffee.assemble(ADVDIFF, 1, TET, *args, tune=coffee.FLAG_CUDA_CORES))
    assert all(torch.equal(g, w) for g, w in zip(torch.autograd.grad(out, [x, cf], d), want))
