"""Stored-operator smoothers through the TMA-fed kernel, asked for: these grids
have 672 and 717 planned tiles, fewer than the default takes (22 per SM).  Ragged
last slice; a 512-wide grid whose +-nx offsets share one window.  Every spec
against the oracle and, bit for bit, against the direct kernel, from zero and
from a given start."""
import numpy as np
import pytest

from oracle.amg import OracleAMG
from oracle.smoother import SmootherSpec, l1_diag, smooth
from paper_2407_09848_gb300 import problems as pr
from parity import assert_parity

pytestmark = pytest.mark.gpu
TOL = 1e-12  # of every FP64 smoother application
GRIDS = {"varcoef81": lambda: pr.varcoef(81, 1.0, 4.0, seed=5, ny=72, nz=63),
         "poisson512": lambda: pr.poisson(512, 24, 28)}
WEIGHTS = [1.2, 0.8, 1.1, 1.4]
SPECS = [("cheb4_opt", 2), ("cheb4_opt", 3), ("cheb4_opt", 4), ("cheb4_opt", 5), ("cheb4_opt", 16),
         ("cheb4", 3), ("weights", 3), ("weights", 4), ("cheb1", 2), ("cheb1_opt", 3),
         ("l1jacobi", 2), ("l1jacobi", 5)]


@pytest.fixture(scope="module", params=sorted(GRIDS))
def case(request):
    from paper_2407_09848_gb300.amgps import Solver, tma_plan_stats
    H = pr.build_hierarchy(GRIDS[request.param](), coarse_max=512)
    tiles = tma_plan_stats(H.levels[0].A, "f64")[0]
    assert 600 < tiles < 22 * 152
    S = Solver().load(H.A, H.P)
    yield H, S
    S.close()


def _set(S, kind, k):
    from paper_2407_09848_gb300.amgps import opt4_weights
    w = WEIGHTS[:k] if kind == "weights" else None
    rho = 1.05 if kind == "cheb1" else 0.0
    S.set_smoother(-1, kind, k, weights=w, rho=rho)
    beta = np.array(w) if w else (opt4_weights(k) if kind == "cheb4_opt" else None)
    return SmootherSpec(kind, k, beta=beta, rho=rho) if rho else SmootherSpec(kind, k, beta=beta)


@pytest.mark.parametrize("kind,k", SPECS, ids=lambda v: str(v))
def test_tma_operators_match_oracle_and_direct(case, kind, k):
    import torch
    H, S = case
    A = H.levels[0].A
    n = A.shape[0]
    g = np.random.default_rng(7 + k)
    b, x0 = g.uniform(-1, 1, n), g.uniform(-1, 1, n)
    bd = torch.from_numpy(b).cuda()
    spec = _set(S, kind, k)
    M = l1_diag(A)
    for zero in (True, False):
        out = []
        for tma in ("always", False):
            S.set_tma(tma)
            x = torch.from_numpy(x0).cuda()
            S.smooth(0, kind, k, bd, x, x_is_zero=zero)
            out.append(x)
        S.synchronize()
        assert torch.equal(out[0], out[1]), zero
        assert_parity(out[0].cpu().numpy(), smooth(A, b, None if zero else x0, spec, M=M), TOL, zero)


def test_tma_cycle_matches_oracle(case):
    import torch
    H, S = case
    n = H.A[0].shape[0]
    spec = _set(S, "cheb4_opt", 4)
    S.set_tma("always")
    r = np.random.default_rng(21).uniform(-1, 1, n)
    z = torch.empty(n, dtype=torch.float64, device="cuda")
    S.vcycle(torch.from_numpy(r).cuda(), z)
    assert_parity(z.cpu().numpy(), OracleAMG(H.A, H.P, spec).vcycle(r), TOL)
