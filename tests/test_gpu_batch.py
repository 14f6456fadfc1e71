"""Batched vectors (loss gradient, error cycles) against the same calls one
vector at a time: a call with m = 1 takes the unbatched path."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2407_09848_gb300 import problems as pr

pytestmark = pytest.mark.gpu


def _wide_spd(n, seed):
    """SPD matrix with scattered rows (explicit slices, not 7 wide) and pair aggregates."""
    g = np.random.default_rng(seed)
    B = sp.random(n, n, density=5.0 / n, random_state=seed, format="csr")
    A = sp.csr_matrix(B + B.T)
    A = sp.csr_matrix(A + sp.diags(np.asarray(abs(A).sum(axis=1)).ravel() + 0.1 + g.random(n)))
    As, Ps = [A], []
    while As[-1].shape[0] > 512:
        m = As[-1].shape[0]
        agg = np.arange(m) // 2
        P = sp.csr_matrix((np.ones(m), agg, np.arange(m + 1)), shape=(m, int(agg[-1]) + 1))
        Ps.append(P)
        As.append(sp.csr_matrix(P.T @ As[-1] @ P))
    return As, Ps


def _load(which):
    from paper_2407_09848_gb300.amgps import Solver
    if which == "wide":
        As, Ps = _wide_spd(1501, 3)
    else:
        H = pr.build_hierarchy(pr.varcoef(which[0], 1.0, 4.0, seed=2, ny=which[1], nz=which[2]), 512)
        As, Ps = H.A, H.P
    return Solver().load(As, Ps), As[0].shape[0]


# 13x11x9: slices with rows past the end; 57x51x48: stored-operator steps on
# level 0 (131,072 rows and more); wide: rows that are not seven entries long
@pytest.mark.parametrize("which", [(13, 11, 9), (57, 51, 48), "wide"])
@pytest.mark.parametrize("m", [2, 5, 33])
def test_batch_equals_single_vectors(which, m):
    import torch
    S, n = _load(which)
    E = torch.from_numpy(pr.vec_normal(n, seed=1, count=m)).cuda()
    one = E.clone()
    S.error_cycles(E, 2)
    for i in range(m):
        S.error_cycles(one[i:i + 1], 2)
    # every vector's operations are the same, in the same order
    assert torch.equal(E, one)
    loss, gw = S.loss_grad(E)
    parts = [S.loss_grad(E[i:i + 1].contiguous()) for i in range(m)]
    # only the order of the sums over the vectors differs
    assert abs(loss - np.mean([p[0] for p in parts])) <= 1e-13 * loss
    ref = np.mean([p[1] for p in parts], axis=0)
    assert np.max(np.abs(gw - ref)) <= 1e-11 * np.max(np.abs(ref))
    S.close()


def test_batch_gives_way_to_the_allocation_limit():
    """A limit that leaves room for the one-vector buffers only: the calls run, same results."""
    import torch
    S, n = _load((57, 51, 48))
    E = torch.from_numpy(pr.vec_normal(n, seed=1, count=9)).cuda()
    free = S.loss_grad(E)
    S.close()
    S, n = _load((57, 51, 48))
    one = S.loss_grad(E[:1].contiguous())        # takes the one-vector buffers
    S.set_alloc_limit(1)                         # nothing more from here on
    lim = S.loss_grad(E)
    assert abs(free[0] - lim[0]) <= 1e-13 * free[0]
    assert np.max(np.abs(free[1] - lim[1])) <= 1e-11 * np.max(np.abs(free[1]))
    assert np.isfinite(one[0])
    S.close()
