"""Which float64 kernels run: products on the integer pipe for coefficients
within 2^-150 .. 2^150 (k in every cell), float64 arithmetic otherwise.

Float64 arithmetic gives the one-point-per-thread kernels' bits; the fixed-point
sums round elsewhere, so that a random field's results differ."""
import numpy as np
import pytest
import torch

import mg_inputs as mi

pytestmark = pytest.mark.gpu


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def field(dims, lowest=None, highest=None):
    """Powers of two around 1, in one cell the lowest or highest value asked for."""
    k = np.exp2(np.round(mi.cell_log10_k(dims, 2, -2.0, 2.0, 83)))
    if lowest is not None:
        k[1, 2, 3] = lowest
    if highest is not None:
        k[2, 1, 0] = highest
    return k


LOW, HIGH = 2.0 ** -150, 2.0 ** 150


@pytest.mark.parametrize("dims", [(9, 17, 33), (17, 25, 137), (41, 49, 65)])
@pytest.mark.parametrize("k,fixed_point", [
    (dict(), True), (dict(lowest=LOW), True), (dict(highest=HIGH), True),
    (dict(lowest=np.nextafter(LOW, 0)), False), (dict(highest=np.nextafter(HIGH, np.inf)), False), (None, False)],
    ids=["ordinary", "lowest", "highest", "below", "above", "scaled"])
def test_kernels_by_coefficient_range(gpu_lib, dims, k, fixed_point):
    mg = gpu_lib
    kc = T(np.ldexp(field(dims), -200) if k is None else field(dims, **k))
    A, B = (mg.MGSolver(kc, mg.Params(stencil_kernel=s, telescope_max_n=0)) for s in (0, 2))
    x, b = T(mi.random_nodal(dims, 84)), T(mi.random_nodal(dims, 85))
    pairs = [(A.smooth(b, x), B.smooth(b, x)), (A.residual_restrict(b, x), B.residual_restrict(b, x))]
    for level in (-1, 0):
        pairs.append((A.apply(x, level), B.apply(x, level)))
    pairs.append((A.vcycle(b), B.vcycle(b)))
    for got, ref in pairs:
        assert torch.equal(got, ref) != fixed_point
    for degree in (1, 3):
        C, D = (mg.MGSolver(kc, mg.Params(stencil_kernel=s, telescope_max_n=0, cheby_degree=degree)) for s in (0, 2))
        assert torch.equal(C.smooth(b, x), D.smooth(b, x)) != fixed_point
        C.close()
        D.close()
    A.close()
    B.close()
