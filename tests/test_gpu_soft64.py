"""The float64 stencil passes with products on the integer pipe, over the
operands they accept: magnitudes that differ by hundreds of binary orders, zeros,
subnormals, values near the float64 limits, and non-finite ones.

Reference: the arithmetic-mean operator in numpy's extended precision.
Tolerance: a point's seven products (coefficients rounded three times, the
diagonal a sum of six) and its sum of seven terms are each off by at most
2^-53 of the terms' absolute sum T, 16 of them in all; 2^-49 T bounds them."""
import numpy as np
import pytest
import torch

import mg_inputs as mi

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def reference(k, x):
    """(A x, sum of the terms' absolute values) at interior nodes, arithmetic edge means, extended precision."""
    k, x = k.astype(np.longdouble), x.astype(np.longdouble)
    n = [s + 1 for s in k.shape]
    y = np.zeros(n, np.longdouble)
    t = np.zeros(n, np.longdouble)
    inner = (slice(1, -1),) * 3
    for a in range(3):
        p, q = [d for d in range(3) if d != a]
        c = k
        for d in (p, q):
            m = c.shape[d] - 1
            c = c.take(range(m), d) + c.take(range(1, m + 1), d)
        c = c / 4 * np.longdouble(n[a] - 1) ** 2
        m = n[a] - 2
        lo, hi = c.take(range(m), a), c.take(range(1, m + 1), a)
        sl = [slice(1, -1)] * 3
        sl[a] = slice(0, -2)
        xl = x[tuple(sl)]
        sl[a] = slice(2, None)
        xh = x[tuple(sl)]
        y[inner] += (lo + hi) * x[inner] - lo * xl - hi * xh
        t[inner] += (lo + hi) * abs(x[inner]) + lo * abs(xl) + hi * abs(xh)
    return y, t


def operand(kind, dims, seed):
    x = mi.random_nodal(dims, seed)
    r = np.random.default_rng(seed)
    inner = (slice(1, -1),) * 3
    shape = x[inner].shape
    if kind == "sparse":
        x[inner] *= r.random(shape) < 0.02
    elif kind == "spread":
        x[inner] = np.ldexp(x[inner], r.integers(-300, 300, shape))
    elif kind == "subnormal":
        x[inner] = np.ldexp(x[inner], r.integers(-1080, -1000, shape))
    elif kind == "huge":
        x[inner] = np.ldexp(x[inner], 990)
    elif kind == "smooth":  # neighbours nearly equal: the sum cancels
        x[inner] = 1.0 + 1e-12 * x[inner]
    return x


@pytest.mark.parametrize("dims", [(3, 3, 3), (5, 9, 33), (17, 33, 97), (41, 49, 129)])
@pytest.mark.parametrize("kind", ["random", "sparse", "spread", "subnormal", "huge", "smooth"])
def test_operator_over_operand_ranges(gpu_lib, dims, kind):
    mg = gpu_lib
    k = mi.cell_k(dims, 2, -2.0, 2.0, 31)
    x = operand(kind, dims, 32)
    ref, t = reference(k, x)
    S = mg.MGSolver(T(k), mg.Params(face_rule=1))
    y = S.apply(T(x), -1)
    err = abs(y.cpu().numpy().astype(np.longdouble) - ref)
    assert np.all(err <= np.ldexp(t, -49) + 16 * np.ldexp(np.longdouble(1), -1074))
    # the padded level's kernel (an input that is also the output) gives the same numbers
    from paper_1604_07163_gb300 import _lib
    buf = T(x)
    assert _lib.load().mg_apply(S._h, -1, buf.data_ptr(), buf.data_ptr()) == 0
    assert torch.equal(buf, y)
    S.close()


def test_non_finite_operands_reach_their_neighbours(gpu_lib):
    mg = gpu_lib
    dims = (9, 17, 33)
    k = mi.cell_k(dims, 2, -1.0, 1.0, 41)
    x = mi.random_nodal(dims, 42)
    x[4, 8, 16], x[2, 3, 5] = np.inf, np.nan
    y = mg.MGSolver(T(k), mg.Params(face_rule=1)).apply(T(x), -1).cpu().numpy()
    hit = np.zeros(dims, bool)
    for p in ((4, 8, 16), (2, 3, 5)):
        for a in range(3):
            for s in (-1, 0, 1):
                q = list(p)
                q[a] += s
                hit[tuple(q)] = True
    assert np.array_equal(~np.isfinite(y), hit)
    assert np.isnan(y[2, 3, 5]) and y[4, 8, 16] == np.inf and y[4, 8, 15] == -np.inf


@pytest.mark.parametrize("dims", [(17, 33, 49), (65, 65, 65)])
def test_out_of_range_coefficients_scale_the_solution(gpu_lib, dims):
    """k times 2^-200 lies outside the coefficients' range, so float64 arithmetic runs: V-cycle and solution are those
    of k scaled by 2^200, but for rounding (1e-12 of the largest value: a V-cycle's and a dozen CG steps' of 1e-16)."""
    mg = gpu_lib
    k = mi.cell_k(dims, 4, -1.0, 1.0, 51)
    f = T(mi.random_nodal(dims, 52))
    A, B = mg.MGSolver(T(k)), mg.MGSolver(T(np.ldexp(k, -200)))
    for a, b in ((A.vcycle(f), B.vcycle(f)), (A.solve(f, 1e-10)[0], B.solve(f, 1e-10)[0])):
        b = torch.ldexp(b, torch.tensor(-200, device=DEV))
        assert ((a - b).abs().max() / a.abs().max()).item() < 1e-12
