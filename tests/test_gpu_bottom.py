"""The bottom kernel in shared memory: levels whose shapes do not split evenly
over its blocks, blocks without a plane on the coarser levels, coarsest levels
of more than 32 unknowns (one product with the inverse, rows over all blocks),
and every form of the sweep.

Tolerances as in the other parity tests: a V-cycle 1e-12 relative to the
largest magnitude; block counts and the global-memory bottom kernel (chosen by
a bottom that does not fit shared memory) bit for bit."""
import numpy as np
import pytest
import torch

import mg_inputs as mi
from test_gpu_parity import N, T, make, relmax

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(9, 9, 17), (13, 21, 29), (25, 17, 41), (33, 9, 9), (9, 33, 9), (5, 33, 9), (3, 5, 9)])
@pytest.mark.parametrize("params", [
    {}, dict(cheby_degree=1), dict(cheby_degree=3, nu_pre=2), dict(nu_pre=0), dict(nu_post=0),
    dict(smoother="richardson", nu_pre=2, nu_post=3), dict(coarse_op="galerkin"), dict(bottom_blocks=1),
    dict(bottom_blocks=2)], ids=str)
def test_bottom_vcycle_and_coarse_solve_match_the_oracle(gpu_lib, dims, params):
    oparams = {k: v for k, v in params.items() if k != "bottom_blocks"}
    k, O, S = make(dims, 2, 2.0, params) if oparams == params else make_blocks(dims, oparams, params)
    r = mi.random_nodal(dims, 61)
    assert relmax(N(S.vcycle(T(r))), O.vcycle(r)) < 1e-12
    bc = mi.random_nodal(O.level_dims(O.levels - 1), 62)
    assert relmax(N(S.coarse_solve(T(bc))), O.coarse_solve(bc)) < 1e-12
    S.close()


def make_blocks(dims, oparams, params):
    import paper_1604_07163_gb300 as mg
    k, O, S = make(dims, 2, 2.0, oparams)
    S.close()
    return k, O, mg.MGSolver(T(k), mg.Params(**params))


@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32", "mixed_bf16k"])
@pytest.mark.parametrize("coarse_op", ["rediscretised", "galerkin"])
def test_global_memory_bottom_gives_the_same_bits(gpu_lib, precision, coarse_op):
    """33 x 41 x 49 with every level in the bottom kernel does not fit shared
    memory; the default split does."""
    import paper_1604_07163_gb300 as mg
    dims = (33, 41, 49)
    k, r = T(mi.cell_k(dims, 4, -2.0, 2.0, 63)), T(mi.random_nodal(dims, 64))
    out = []
    for tele in (4096, 1 << 20):
        S = mg.MGSolver(k, mg.Params(precision=precision, coarse_op=coarse_op, telescope_max_n=tele, stencil_kernel=2))
        out.append(S.vcycle(r))
        S.close()
    assert torch.equal(out[0], out[1])
