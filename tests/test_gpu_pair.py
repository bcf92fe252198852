"""Two smoothing passes in one sweep give the single passes' V-cycle bit for bit
(the one-point-per-thread driver runs them singly): one tile per row and rows
wider than a tile, odd and even numbers of steps, ends of plane chunks."""
import numpy as np
import pytest
import torch

import mg_inputs as mi

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


@pytest.mark.parametrize("dims", [(161, 161, 161), (129, 129, 513), (513, 161, 65)])
@pytest.mark.parametrize("kw", [dict(), dict(precision="mixed_bf16k"), dict(nu_post=2),
                                dict(smoother="richardson", nu_pre=1, nu_post=2),
                                dict(smoother="richardson", nu_pre=3, nu_post=1),
                                dict(smoother="richardson", nu_pre=4, nu_post=3)], ids=str)
def test_vcycle(gpu_lib, dims, kw):
    mg = gpu_lib
    kw = dict(dict(precision="mixed_fp32"), **kw)
    k = T(mi.cell_k(dims, 8, -2.0, 2.0, 81))
    r = T(mi.random_nodal(dims, 82))
    z = [mg.MGSolver(k, mg.Params(stencil_kernel=s, **kw)).vcycle(r) for s in (0, 2)]
    assert z[0].abs().max().item() > 0
    assert torch.equal(z[0], z[1])


def test_solve_forms_the_same_rho(gpu_lib):
    """rho = b.z is summed in another grouping: iterates agree to rounding (1e-10 of the largest value, the tolerance of the solve)."""
    mg = gpu_lib
    dims = (161, 161, 161)
    k, f = T(mi.cell_k(dims, 8, -1.0, 1.0, 83)), T(mi.random_nodal(dims, 84))
    (x, s), (y, t) = (mg.MGSolver(k, mg.Params(precision="mixed_fp32", face_rule=1, stencil_kernel=s)).solve(f, 1e-10)
                      for s in (0, 2))
    assert s.iters == t.iters
    assert ((x - y).abs().max() / y.abs().max()).item() < 1e-10
