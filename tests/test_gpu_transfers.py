"""The vector kernels of the transfers, of the float32 7-point passes and of the
27-point passes give the one-point-per-thread kernels' results bit for bit: rows that end inside a
vector, rows wider than a warp's, level sizes down to three points."""
import numpy as np
import pytest
import torch

import mg_inputs as mi

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
DIMS = [(9, 9, 9), (17, 9, 25), (33, 17, 73), (17, 25, 265), (33, 33, 529), (41, 49, 129)]


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def pair(mg, dims, **kw):
    k = T(mi.cell_k(dims, 2, -2.0, 2.0, 61))
    return [mg.MGSolver(k, mg.Params(stencil_kernel=s, telescope_max_n=0, **kw)) for s in (0, 2)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32"])
def test_transfers(gpu_lib, dims, precision):
    A, B = pair(gpu_lib, dims, precision=precision)
    for l in range(A.num_levels - 1):
        shape, coarse = A.level_shape(l), A.level_shape(l + 1)
        x, b, e = (T(mi.random_nodal(s, 62 + i)) for i, s in enumerate((shape, shape, coarse)))
        assert torch.equal(A.prolong_add(e, x, l), B.prolong_add(e, x, l))
        if precision != "fp64":  # in float64 the residuals differ in rounding
            assert torch.equal(A.residual_restrict(b, x, l), B.residual_restrict(b, x, l))
        # the restriction alone: with x = 0 the residual is b in either kernel
        z = torch.zeros_like(x)
        assert torch.equal(A.residual_restrict(b, z, l), B.residual_restrict(b, z, l))


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("precision", ["mixed_fp32", "mixed_bf16k"])
@pytest.mark.parametrize("degree", [2, 3])
def test_7_point_smoothing(gpu_lib, dims, precision, degree):
    A, B = pair(gpu_lib, dims, precision=precision, cheby_degree=degree)
    for l in range(A.num_levels):
        b, x = (T(mi.random_nodal(A.level_shape(l), 66 + i)) for i in range(2))
        assert torch.equal(A.smooth(b, None, l), B.smooth(b, None, l))
        assert torch.equal(A.smooth(b, x, l), B.smooth(b, x, l))


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32", "mixed_bf16k"])
@pytest.mark.parametrize("degree", [2, 3])
def test_27_point_passes(gpu_lib, dims, precision, degree):
    A, B = pair(gpu_lib, dims, precision=precision, coarse_op="galerkin", cheby_degree=degree)
    for l in range(1, A.num_levels):
        b, x = (T(mi.random_nodal(A.level_shape(l), 71 + i)) for i in range(2))
        assert torch.equal(A.smooth(b, None, l), B.smooth(b, None, l))
        assert torch.equal(A.smooth(b, x, l), B.smooth(b, x, l))
        if l + 1 < A.num_levels:
            assert torch.equal(A.residual_restrict(b, x, l), B.residual_restrict(b, x, l))
