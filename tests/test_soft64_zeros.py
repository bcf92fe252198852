"""The float64 stencil passes on zero operands, which the fixed-point products
leave to float64 arithmetic: signs, and time."""
import numpy as np
import pytest
import torch

import mg_inputs as mi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(5, 9, 33), (17, 33, 97)])
def test_operator_on_signed_zeros(gpu_lib, dims):
    """Zeros of either sign: the signs of float64 arithmetic, in both of the operator's kernels."""
    mg = gpu_lib
    k = torch.tensor(mi.cell_k(dims, 2, -2.0, 2.0, 95), device="cuda:0")
    x = np.copysign(0.0, mi.random_nodal(dims, 96))
    x[2, 2:6, 2:20] = -0.0
    x = torch.tensor(x, device="cuda:0")
    A, B = (mg.MGSolver(k, mg.Params(stencil_kernel=s)) for s in (0, 2))
    y, ref = A.apply(x, -1), B.apply(x, -1)
    assert torch.equal(y, torch.zeros_like(y)) and torch.equal(torch.signbit(y), torch.signbit(ref))
    from paper_1604_07163_gb300 import _lib
    buf = x.clone()
    assert _lib.load().mg_apply(A._h, -1, buf.data_ptr(), buf.data_ptr()) == 0
    assert torch.equal(torch.signbit(buf), torch.signbit(y))


def test_zeros_take_little_longer_than_other_operands(gpu_lib):
    """A V-cycle on a field that vanishes: with the whole sum formed again at every point it took 1.5 times as long."""
    mg = gpu_lib
    dims = (257, 257, 257)
    S = mg.MGSolver(torch.tensor(mi.cell_k(dims, 16, -2.0, 2.0, 97), device="cuda:0"))
    x = torch.tensor(mi.random_nodal(dims, 98), device="cuda:0")
    best = []
    for v in (x, torch.zeros_like(x)):
        times = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            S.vcycle(v)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        best.append(min(times[2:]))
    assert best[1] < 1.35 * best[0]
