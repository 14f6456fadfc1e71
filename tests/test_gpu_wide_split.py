"""Warps per slice of wide rows: the rules for waves that are not full and for a
slice much wider than the rest, and the split step's batches on uniform slices
(remainders, slices narrower than a batch), against the oracle."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle.smoother import SmootherSpec, l1_diag, smooth

pytestmark = pytest.mark.gpu


def _spd(off, g):
    off = sp.csr_matrix(off + off.T)
    n = off.shape[0]
    return sp.csr_matrix(off + sp.diags(np.asarray(abs(off).sum(axis=1)).ravel() + 0.1 + g.random(n)))


def _band(n, half, g):
    return sp.diags([-(0.5 + g.random(n - o)) for o in range(1, half + 1)],
                    list(range(1, half + 1)), shape=(n, n), format="csr")


def _matrix(which):
    g = np.random.default_rng(3)
    if which == "band":        # 313 slices of 251, 8 warps: 31 or 32 entries a warp
        return _spd(_band(10005, 125, g), g)
    if which == "unfilled":    # 626 slices of 501: 16 warps instead of 4
        return _spd(_band(20005, 250, g), g)
    if which == "narrow":      # slices of 5 and of 101 entries, 4 warps
        return _spd(sp.block_diag([_band(6400, 2, g), _band(6001, 50, g)], format="csr"), g)
    n = 20005                  # "dense": 81 entries a row, one row of 2,000
    B = sp.lil_matrix(_band(n, 40, g))
    B[0, 41:2040] = -0.01
    return _spd(sp.csr_matrix(B), g)


@pytest.mark.parametrize("which", ["band", "unfilled", "narrow", "dense"])
def test_split_rows_equal_oracle(which):
    import torch
    from paper_2407_09848_gb300.amgps import Solver
    A = _matrix(which)
    n = A.shape[0]
    nc = 500
    P = sp.csr_matrix((np.ones(n), (np.arange(n) * nc) // n, np.arange(n + 1)), shape=(n, nc))
    Ac = sp.csr_matrix(P.T @ A @ P)
    g = np.random.default_rng(4)
    b, x0 = g.uniform(-1, 1, n), g.uniform(-1, 1, n)
    M = l1_diag(A)
    w = int(np.diff(A.indptr).max())
    for prec in ("f64", "f32"):
        S = Solver().load([A, Ac], [P], prec=prec)
        for kind, k in [("cheb4", 3), ("cheb1_opt", 2), ("l1jacobi", 2)]:
            x = torch.from_numpy(x0).cuda()
            S.smooth(0, kind, k, torch.from_numpy(b).cuda(), x)
            ref = smooth(A, b, x0, SmootherSpec(kind, k), M=M)
            # FP32: every step sums rows of M^-1 A, whose entries add up to 1
            tol = 1e-12 if prec == "f64" else k * (w + 3) * 2.0 ** -24
            err = np.linalg.norm(x.cpu().numpy() - ref)
            assert err <= tol * (np.linalg.norm(ref) + np.linalg.norm(x0)), (prec, kind, k)
        S.close()
