"""Coarse l1-Jacobi sweeps as one matrix against the sweeps themselves (which
run when the allocation limit leaves no room for the matrix)."""
import numpy as np
import pytest

from paper_2407_09848_gb300 import problems as pr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,coarse_max", [((5, 5, 5), 4), ((13, 11, 9), 512), ((24, 20, 18), 1024)])
@pytest.mark.parametrize("m", [3, 4, 30])
def test_sweep_matrix_equals_sweeps(shape, coarse_max, m):
    import torch
    from paper_2407_09848_gb300.amgps import Solver
    H = pr.build_hierarchy(pr.varcoef(shape[0], 1.0, 4.0, seed=4, ny=shape[1], nz=shape[2]),
                           coarse_max)
    n = H.A[0].shape[0]
    r = torch.from_numpy(pr.rhs_uniform(n, seed=1)).cuda()
    z = [torch.empty_like(r) for _ in range(2)]
    for i in range(2):
        S = Solver().load(H.A, H.P)
        if i:
            S.set_alloc_limit(1)
        S.set_coarse_sweeps(m)
        S.vcycle(r, z[i])
        torch.cuda.synchronize()
        S.close()
    # m sweeps of at most 1024-term sums against one such sum
    assert torch.linalg.norm(z[0] - z[1]) <= 1e-13 * torch.linalg.norm(z[1])
