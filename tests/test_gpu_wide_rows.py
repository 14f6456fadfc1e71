"""Wide rows on FP64 levels (several lanes and warps per row) against the
oracle: every split, ragged last slices, widths that leave lanes idle."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle.amg import OracleAMG
from oracle.smoother import SmootherSpec
from paper_2407_09848_gb300 import problems as pr

pytestmark = pytest.mark.gpu


def _matrix(n, half, scattered, seed):
    """Symmetric, 2 half + 1 entries a row: a band (uniform slices) or the band
    under a permutation (explicit slices)."""
    g = np.random.default_rng(seed)
    offs = range(1, half + 1)
    d = [-(0.5 + g.random(n - o)) for o in offs]
    A = sp.diags(d, list(offs), shape=(n, n), format="csr")
    A = sp.csr_matrix(A + A.T)
    A = sp.csr_matrix(A + sp.diags(np.asarray(abs(A).sum(axis=1)).ravel() + 0.1 + g.random(n)))
    if scattered:
        p = g.permutation(n)
        A = sp.csr_matrix(A[p][:, p])
    return A


def _smoothed(A, n):
    """A prolongator with several entries a row (general transfers)."""
    agg = np.arange(n) // 9
    Ph = sp.csr_matrix((np.ones(n), agg, np.arange(n + 1)), shape=(n, int(agg[-1]) + 1))
    return sp.csr_matrix(Ph - 0.3 * sp.diags(1.0 / A.diagonal()) @ (A @ Ph))


# 2 half + 1 entries on n rows: splits 2, 4, 8, 16 and 32 (warps per slice)
@pytest.mark.parametrize("n,half", [(8197, 12), (1999, 17), (2010, 33), (1030, 70), (1300, 130)])
@pytest.mark.parametrize("scattered", [False, True])
def test_wide_rows_equal_oracle(n, half, scattered):
    import torch
    from paper_2407_09848_gb300.amgps import Solver
    A = _matrix(n, half, scattered, 1)
    P = _smoothed(_matrix(n, half, False, 1), n)
    As, Ps = [A, sp.csr_matrix(P.T @ A @ P)], [P]
    S = Solver().load(As, Ps)
    r = pr.rhs_uniform(n, seed=2)
    rd = torch.from_numpy(r).cuda()
    z = torch.empty_like(rd)
    for kind, k in [("cheb4_opt", 4), ("cheb1_opt", 3), ("l1jacobi", 2)]:
        S.set_smoother(-1, kind, k)
        S.vcycle(rd, z)
        ref = OracleAMG(As, Ps, SmootherSpec(kind, k)).vcycle(r)
        assert np.linalg.norm(z.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref), (kind, k)
    S.close()
