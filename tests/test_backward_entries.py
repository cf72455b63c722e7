"""FP64 adjoint, factor by factor: on cells that are scaled reference cells the gradient of the advection velocity at
vertex v is h^(d-1) Gbar[v][a], one factor's sum_o T[k][o] dA[o] each, to rounding of its own terms also where other
entries of dA are far larger (a dominant entry, entries of very different size, one row alone).

Tolerance against the plain kernel (FLAG_CUDA_CORES), of sum_o |T[k][o] dA[o]|: N roundings there; by digits a step of
2^-55 of the scale, of which an entry above 2^-4 and a T above 2^-2 leave 2^-8 or more with the exponents' slack of
2^-1 in all, 64 roundings; cells without such entries are summed as the plain kernel sums them. (N + 64) 2^-53."""
import numpy as np
import pytest
import torch

import paper_1407_0904_gb300 as coffee
from tests.helpers import TRI, TET, ADVDIFF, FP64
from tests.test_backward_tc import backward

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("cell,k", [(TRI, 1), (TRI, 2), (TRI, 4), (TET, 1), (TET, 2), (TET, 3)])
@pytest.mark.parametrize("kind", ["even", "dominant", "spread", "row"])
def test_velocity_gradients_to_rounding_of_their_terms(cell, k, kind):
    rng = np.random.default_rng(3)
    d, nc = 2 if cell == TRI else 3, 150
    h = 2.0 ** rng.integers(-3, 3, nc)
    ref = np.concatenate([np.zeros((1, d)), np.eye(d)])
    coords = (h[:, None, None] * ref).reshape(-1, d)
    c2v = np.arange(nc * (d + 1), dtype=np.int32).reshape(nc, d + 1)
    coef = rng.random(nc * (d + 1) * (d + 1))
    T = np.asarray(coffee.reference_tensor(ADVDIFF, k, cell))
    N = T.reshape(T.shape[0], -1).shape[1]
    n = round(N ** 0.5)
    dA = rng.standard_normal((nc, N))
    if kind == "dominant":
        dA[np.arange(nc), rng.integers(0, N, nc)] *= 1e12
    elif kind == "spread":
        dA *= np.exp(rng.uniform(-20, 20, dA.shape))
    elif kind == "row":
        keep = np.zeros((nc, n, n))
        keep[np.arange(nc), rng.integers(0, n, nc)] = 1.0
        dA *= keep.reshape(nc, N)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    args, dout = [t(coords), t(c2v), t(coef), t(c2v)], t(dA.reshape(nc, n, n))
    got, want = (backward(ADVDIFF, k, cell, args, dout, f)[1].view(nc, d + 1, d + 1)[:, :, 1:].cpu().numpy()
                 for f in (0, coffee.FLAG_CUDA_CORES))
    adv = np.abs(T.reshape(T.shape[0], -1)[-(d + 1) * d:])
    size = (np.abs(dA) @ adv.T).reshape(nc, d + 1, d) * h[:, None, None] ** (d - 1)
    assert np.all(np.abs(got - want) <= (N + 64) * 2.0 ** -53 * size)
