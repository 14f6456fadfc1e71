"""Which levels restrict in one kernel: those whose longest aggregate takes at
most two rounds of eight lanes.  On both sides of that line the results are
those of the separate kernels (which run when the coarse levels are recorded for
the cooperative kernel)."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2407_09848_gb300 import problems as pr
from paper_2407_09848_gb300.amgps import PROF_COUNT

pytestmark = pytest.mark.gpu


def _chain(n, longest, seed):
    """A chain, three levels, aggregates of 1 to `longest` rows, the last of `longest`."""
    g = np.random.default_rng(seed)
    A = sp.diags([-np.ones(n - 1), 2.2 + g.random(n), -np.ones(n - 1)], [-1, 0, 1], format="csr")
    As, Ps = [sp.csr_matrix(A)], []
    for _ in range(2):
        m = As[-1].shape[0]
        sizes = [longest]
        while sum(sizes) < m:
            sizes.insert(0, int(min(m - sum(sizes), g.integers(1, longest + 1))))
        agg = np.repeat(np.arange(len(sizes)), sizes)
        P = sp.csr_matrix((np.ones(m), agg, np.arange(m + 1)), shape=(m, len(sizes)))
        Ps.append(P)
        As.append(sp.csr_matrix(P.T @ As[-1] @ P))
    return As, Ps


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("kind,k", [("cheb4_opt", 4), ("cheb1_opt", 3), ("l1jacobi", 2), ("cheb4", 1)])
def test_one_kernel_up_to_two_rounds(prec, kind, k):
    import torch
    from paper_2407_09848_gb300.amgps import Solver
    count = {}
    for longest in (9, 16, 17):
        As, Ps = _chain(4003, longest, 1)
        S = Solver().load(As, Ps, prec=prec)
        S.set_smoother(-1, kind, k)
        r = torch.from_numpy(pr.rhs_uniform(4003, seed=1)).cuda()
        z, y = torch.empty_like(r), torch.empty_like(r)
        S.vcycle(r, z)
        S.profile_read(PROF_COUNT, reset=True)
        S.vcycle(r, z)
        count[longest] = S.profile_read(PROF_COUNT, reset=True)[0]
        S.set_coarse_kernel(True)
        S.vcycle(r, y)
        S.synchronize()
        assert torch.equal(z, y)
        S.close()
    assert count[9] == count[16]
    assert count[17] >= count[16] + 2  # residual and sums apart on either level
