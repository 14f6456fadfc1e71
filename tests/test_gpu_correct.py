"""Coarse correction with the first post-smoothing step (one kernel, four
entries of M^-1 A P a row) against the oracle's V-cycle, and the levels that
keep the prolongation."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle.amg import OracleAMG
from oracle.smoother import SmootherSpec
from paper_2407_09848_gb300 import problems as pr

pytestmark = pytest.mark.gpu


def _check(As, Ps, kind, k, form=1):
    import torch
    from paper_2407_09848_gb300.amgps import Solver
    S = Solver().load(As, Ps)
    S.set_step_form(form)
    S.set_smoother(-1, kind, k)
    r = pr.rhs_uniform(As[0].shape[0], seed=3)
    z = torch.empty(r.size, dtype=torch.float64, device="cuda")
    S.vcycle(torch.from_numpy(r).cuda(), z)
    ref = OracleAMG(As, Ps, SmootherSpec(kind, k)).vcycle(r)
    S.close()
    assert np.linalg.norm(z.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)


# ragged grids: last slices with rows past the end, blocks one cell wide; the
# last one has a level in the stored-operator form (131,072 rows and more)
@pytest.mark.parametrize("shape", [(9, 8, 7), (33, 17, 13), (53, 51, 50)])
@pytest.mark.parametrize("kind", ["cheb4_opt", "cheb1_opt", "l1jacobi"])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 6])
def test_correction_equals_oracle(shape, kind, k):
    H = pr.build_hierarchy(pr.varcoef(shape[0], 1.0, 4.0, seed=5, ny=shape[1], nz=shape[2]), 64)
    _check(H.A, H.P, kind, k)


@pytest.mark.parametrize("k", [2, 4])
def test_correction_with_the_recurrence_form(k):
    H = pr.build_hierarchy(pr.varcoef(53, 1.0, 4.0, seed=5, ny=51, nz=50), 64)
    _check(H.A, H.P, "cheb4_opt", k, form=0)


@pytest.mark.parametrize("far", [(1, 40), (1, 40, 80), (1, 40, 80, 120)])
def test_rows_that_touch_other_numbers_of_aggregates(far):
    """Chains with far couplings, 40 rows an aggregate in shuffled order: rows
    touch 3 aggregates (corrected), 5 (refused while the matrix is formed), or
    are wider than eight entries; the refused levels keep the prolongation."""
    n = 1300
    A = sp.lil_matrix((n, n))
    for o in far:
        i = np.arange(n - o)
        A[i, i + o] = -1.0
        A[i + o, i] = -1.0
    A = sp.csr_matrix(A)
    A = sp.csr_matrix(A + sp.diags(np.asarray(abs(A).sum(axis=1)).ravel() + 0.5))
    agg = np.random.default_rng(0).permutation((n + 39) // 40)[np.arange(n) // 40]
    P = sp.csr_matrix((np.ones(n), agg, np.arange(n + 1)), shape=(n, int(agg.max()) + 1))
    _check([A, sp.csr_matrix(P.T @ A @ P)], [P], "cheb4_opt", 4)
