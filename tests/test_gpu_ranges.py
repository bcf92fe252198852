"""Operands near the ends of the number range: what is finite in the scalar
kernels, or in real arithmetic scaled by a power of two, stays so."""
import numpy as np
import pytest
import torch

import mg_inputs as mi

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


@pytest.mark.parametrize("dims", [(9, 9, 9), (17, 9, 25), (17, 25, 265), (41, 49, 129)])
@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32", "mixed_bf16k"])
def test_restriction_of_large_residuals(gpu_lib, dims, precision):
    """Residuals up to a quarter of the largest number of the V-cycle's type restrict as in the one-point-per-thread
    kernel, bit for bit."""
    mg = gpu_lib
    k = T(mi.cell_k(dims, 2, -2.0, 2.0, 81))
    A, B = (mg.MGSolver(k, mg.Params(stencil_kernel=s, telescope_max_n=0, precision=precision)) for s in (0, 2))
    e = 1022 if precision == "fp64" else 126
    for l in range(A.num_levels - 1):
        b = T(np.ldexp(mi.random_nodal(A.level_shape(l), 82), e))
        z = torch.zeros_like(b)
        got = A.residual_restrict(b, z, l)
        assert bool(torch.isfinite(got).all())
        assert torch.equal(got, B.residual_restrict(b, z, l))
    A.close()
    B.close()


@pytest.mark.parametrize("dims", [(9, 17, 33), (41, 49, 129)])
@pytest.mark.parametrize("face_rule", [0, 1])
@pytest.mark.parametrize("ek,ex", [(500, 0), (400, 160), (-500, -60)])
def test_cell_gradient_scales_with_its_operands(gpu_lib, dims, face_rule, ek, ex):
    """k times 2^ek, phi and lambda times 2^ex: the gradient times 2^(ek + 2 ex), bit for bit (h^-4 k^2 and its products
    with dphi dlambda would leave the range, h^-2 k and the gradient do not)."""
    mg = gpu_lib
    k, x, lam = (mi.cell_k(dims, 2, -1.0, 1.0, 91), mi.random_nodal(dims, 92), mi.random_nodal(dims, 93))
    g = []
    for a, b in ((0, 0), (ek, ex)):
        S = mg.MGSolver(T(np.ldexp(k, a)), mg.Params(face_rule=face_rule))
        g.append(S.gradient(T(np.ldexp(x, b)), T(np.ldexp(lam, b))).cpu().numpy())
        S.close()
    assert np.array_equal(g[1], np.ldexp(g[0], ek + 2 * ex))
