"""A cell gradient written over one of its inputs allocates nothing, so that it can be captured into a CUDA graph."""
import numpy as np
import pytest
import torch

import mg_inputs as mi

pytestmark = pytest.mark.gpu

DIMS = (193, 193, 193)


def T(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


@pytest.fixture
def setup(gpu_lib):
    from paper_1604_07163_gb300 import _lib
    S = gpu_lib.MGSolver(T(mi.cell_k(DIMS, 16, -1.0, 1.0, 25)))
    phi, lam = T(mi.random_nodal(DIMS, 26)), T(mi.random_nodal(DIMS, 27))
    yield _lib.load(), S, phi, lam, S.gradient(phi, lam)
    S.close()


def over(lib, S, phi, buf):
    assert lib.mg_gradient(S._h, phi.data_ptr(), buf.data_ptr(), buf.data_ptr()) == 0


def result(buf, g):
    return buf.reshape(-1)[:g.numel()].reshape(g.shape)


def test_allocates_nothing_and_leaves_the_solver_as_it_was(setup):
    lib, S, phi, lam, g = setup
    x = S.solve(phi, 1e-8)[0]
    buf = lam.clone()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    over(lib, S, phi, buf)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    assert torch.equal(result(buf, g), g)
    assert torch.equal(S.solve(phi, 1e-8)[0], x)


def test_under_capture(setup):
    lib, S, phi, lam, g = setup
    buf = lam.clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        S._sync_stream()
        over(lib, S, phi, buf)
    for _ in range(2):
        buf.copy_(lam)
        graph.replay()
        assert torch.equal(result(buf, g), g)
