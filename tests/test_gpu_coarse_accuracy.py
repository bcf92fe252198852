"""How near the coarsest solve comes to the solution.

The operator is exact in float64 (integer k, arithmetic edge means, h^-2 an
integer), the reference its solution in extended precision.  The solve is a
product with the stored inverse, whose entries are correct to one rounding
(2^-53); with a right-hand side of one sign all terms have one sign, so that a
sum of n/32 multiply-adds and a tree of five additions is off by at most
(n/32 + 5) 2^-53 of itself.  Substitution with a Cholesky factor, or an inverse
formed with it, is off by a multiple of the condition number instead."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def operator(k):
    dims = tuple(s - 1 for s in k.shape)
    n = dims[0] * dims[1] * dims[2]
    A, num = np.zeros((n, n)), np.arange(n).reshape(dims)
    for a in range(3):
        c = k
        for d in range(3):
            if d != a:
                m = c.shape[d] - 1
                c = c.take(range(m), d) + c.take(range(1, m + 1), d)
        c = c / 4 * float(k.shape[a]) ** 2
        m = dims[a]
        for lo in (0, 1):  # the edge below, the edge above
            e = c.take(range(lo, lo + m), a)
            A[num, num] += e
            i = num.take(range(1 - lo, m - lo), a)
            A[i, num.take(range(0, m - 1) if lo == 0 else range(1, m), a)] = -e.take(range(1 - lo, m - lo), a)
    return A


@pytest.mark.parametrize("dims", [(5, 5, 5), (4, 6, 6), (6, 6, 6), (7, 6, 8), (9, 9, 9), (12, 12, 12)])
@pytest.mark.parametrize("bits", [3, 20])
def test_coarse_solve_error(gpu_lib, dims, bits):
    mg = gpu_lib
    rng = np.random.default_rng(7)
    k = np.round(np.exp2(rng.uniform(0, bits, [d - 1 for d in dims])))
    A = operator(k)
    assert np.array_equal(A, A.T)
    n = len(A)
    b = rng.uniform(0.5, 1.0, n)
    x = np.linalg.solve(A, b).astype(np.longdouble)
    for _ in range(8):
        x += np.linalg.solve(A, (b - A.astype(np.longdouble) @ x).astype(float))
    f = np.zeros(dims)
    f[1:-1, 1:-1, 1:-1] = b.reshape([d - 2 for d in dims])
    S = mg.MGSolver(torch.tensor(k, device="cuda:0"), mg.Params(levels=1, face_rule=1))
    got = S.coarse_solve(torch.tensor(f, device="cuda:0")).cpu().numpy()[1:-1, 1:-1, 1:-1].reshape(-1)
    S.close()
    err = np.abs(got.astype(np.longdouble) - x)
    assert np.all(err <= (n / 32 + 8) * np.ldexp(x, -53))
