"""Large levels of wide rows keep the recurrence form (stored operators there
are several copies of a matrix of gigabytes for two of some 170 FP64
instructions a row)."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


def test_wide_large_level_keeps_the_recurrence_form():
    import torch
    from paper_2407_09848_gb300.amgps import AmgpsError, Solver
    n, half = 160000, 25  # 5000 slices of 51 entries
    g = np.random.default_rng(5)
    offs = [o for o in range(-half, half + 1) if o]
    A = sp.diags([np.full(n - abs(o), -1.0 / (1 + abs(o))) for o in offs], offs, format="csr")
    A = sp.csr_matrix(A + sp.diags(np.asarray(abs(A).sum(axis=1)).ravel() + 0.1 + g.random(n)))
    agg = np.arange(n) // 200
    P = sp.csr_matrix((np.ones(n), agg, np.arange(n + 1)), shape=(n, 800))
    S = Solver().load([A, sp.csr_matrix(P.T @ A @ P)], [P])
    b, x0 = (torch.from_numpy(g.uniform(-1, 1, n)).cuda() for _ in range(2))
    out = []
    for form in (1, 0):
        S.set_step_form(form)
        x = x0.clone()
        S.smooth(0, "cheb4_opt", 4, b, x)
        out.append(x)
    S.synchronize()
    assert torch.equal(out[0], out[1])
    S.close()
