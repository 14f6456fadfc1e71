"""Residual, restriction and next level's first step in one kernel (small
levels) against the separate kernels, which run when the coarse levels are
recorded for the cooperative kernel: same bits for every precision."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2407_09848_gb300 import problems as pr

pytestmark = pytest.mark.gpu


def _uneven(n, seed):
    """A chain with aggregates of 1 to 21 rows (lists longer than one round of eight)."""
    g = np.random.default_rng(seed)
    A = sp.diags([-np.ones(n - 1), 2.2 + g.random(n), -np.ones(n - 1)], [-1, 0, 1], format="csr")
    As, Ps = [sp.csr_matrix(A)], []
    for _ in range(2):
        m = As[-1].shape[0]
        sizes = []
        while sum(sizes) < m:
            sizes.append(int(g.integers(1, 22)))
        agg = np.repeat(np.arange(len(sizes)), sizes)[:m]
        P = sp.csr_matrix((np.ones(m), agg, np.arange(m + 1)), shape=(m, int(agg[-1]) + 1))
        Ps.append(P)
        As.append(sp.csr_matrix(P.T @ As[-1] @ P))
    return As, Ps


@pytest.mark.parametrize("which", [(13, 11, 9), (31, 30, 29), "uneven"])
@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("kind,k", [("cheb4_opt", 4), ("cheb1_opt", 3), ("l1jacobi", 2), ("cheb4", 1)])
def test_fused_restriction_equals_separate_kernels(which, prec, kind, k):
    import torch
    from paper_2407_09848_gb300.amgps import Solver
    if which == "uneven":
        As, Ps = _uneven(4003, 1)
    else:
        H = pr.build_hierarchy(pr.varcoef(which[0], 1.0, 4.0, seed=6, ny=which[1], nz=which[2]), 16)
        As, Ps = H.A, H.P
    S = Solver().load(As, Ps, prec=prec)
    S.set_smoother(-1, kind, k)
    r = torch.from_numpy(pr.rhs_uniform(As[0].shape[0], seed=1)).cuda()
    z, y = torch.empty_like(r), torch.empty_like(r)
    S.vcycle(r, z)
    S.set_coarse_kernel(True)
    S.vcycle(r, y)
    S.synchronize()
    assert torch.equal(z, y)
    S.close()
