"""What setup needs only for itself is given back."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_one_matrix_of_the_coarsest_size_is_held(gpu_lib):
    """1000 coarsest unknowns: the inverse takes 8 MB, everything else fits a chunk of 2 MB."""
    mg = gpu_lib
    k = torch.ones((11, 11, 11), dtype=torch.float64, device="cuda:0")
    mg.MGSolver(k, mg.Params(levels=1)).close()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    S = mg.MGSolver(k, mg.Params(levels=1))
    torch.cuda.synchronize()
    held = free - torch.cuda.mem_get_info()[0]
    S.close()
    assert 8e6 <= held <= 14e6
