"""The kernels that work on the caller's dense arrays directly: the float64
operator product and the cell gradient, at the edges of their tiles (32 x 4
nodes; 31 x 4 cells; plane chunks).

Tolerance: as the other float64 steps, a few ulp of the largest term, 1e-13
relative to the largest output magnitude."""
import numpy as np
import pytest
import torch

import mg_inputs as mi
import oracle

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def relmax(a, b):
    return np.max(np.abs(a - b)) / np.max(np.abs(b))


@pytest.mark.parametrize("dims", [(3, 3, 3), (5, 9, 33), (9, 9, 65), (17, 33, 97), (33, 17, 9), (41, 49, 129)])
@pytest.mark.parametrize("face_rule", [0, 1])
def test_dense_operator_and_gradient_match_the_oracle(gpu_lib, dims, face_rule):
    mg = gpu_lib
    k = mi.cell_k(dims, 2, -2.0, 2.0, 11)
    O = oracle.Oracle(k, face_rule=face_rule)
    S = mg.MGSolver(T(k), mg.Params(face_rule=face_rule))
    x, lam = mi.random_nodal(dims, 12), mi.random_nodal(dims, 13)
    junk_x, junk_lam = T(x), T(lam)
    for t in (junk_x, junk_lam):  # boundary entries are ignored whatever they hold
        t[0], t[-1], t[:, 0], t[:, -1], t[:, :, 0], t[:, :, -1] = (float("nan"),) * 6
    for level in (-1, 0):
        assert relmax(S.apply(junk_x, level).cpu().numpy(), O.apply(x)) < 1e-13
    g, go = S.gradient(junk_x, junk_lam).cpu().numpy(), O.gradient(x, lam)
    assert relmax(g, go) < 1e-13
    S.close()


def test_in_place_operator_product_and_overlapping_gradient(gpu_lib):
    """Outputs that overlap an input, through the C ABI."""
    mg = gpu_lib
    from paper_1604_07163_gb300 import _lib
    lib = _lib.load()
    dims = (9, 17, 33)
    k = mi.cell_k(dims, 2, -1.0, 1.0, 21)
    S = mg.MGSolver(T(k))
    x, lam = T(mi.random_nodal(dims, 22)), T(mi.random_nodal(dims, 23))
    y, g = S.apply(x, -1), S.gradient(x, lam)
    buf = x.clone()
    assert lib.mg_apply(S._h, -1, buf.data_ptr(), buf.data_ptr()) == 0
    assert torch.equal(buf, y)
    for a, b in ((x.clone(), lam.clone()), (lam.clone(), x.clone())):  # the gradient over its first, then its second input
        first = b is not None and torch.equal(a, x)
        phi, la = (a, b) if first else (b, a)
        assert lib.mg_gradient(S._h, phi.data_ptr(), la.data_ptr(), a.data_ptr()) == 0
        assert torch.equal(a.reshape(-1)[:g.numel()].reshape(g.shape), g)
    S.close()
