"""Error cycles in several batches, the last of one vector: the graph of the
coarse levels (and the persistent coarse kernel) that an earlier V-cycle has
built belongs to the context's own buffers, not to a batch's; and more vectors
than a grid has blocks in y."""
import pytest

from paper_2407_09848_gb300 import problems as pr
from paper_2407_09848_gb300.amgps import PROF_COUNT

pytestmark = pytest.mark.gpu


def _hierarchy(shape, coarse_max):
    return pr.build_hierarchy(pr.varcoef(shape[0], 1.0, 4.0, seed=2, ny=shape[1], nz=shape[2]),
                              coarse_max)


def _launches(S, f):
    S.profile_read(PROF_COUNT, reset=True)
    f()
    return S.profile_read(PROF_COUNT, reset=True)[0]


def _limit_for_two(H):
    """A limit under which two or three vectors' batch buffers fit, five do not."""
    from paper_2407_09848_gb300.amgps import AmgpsError, Solver
    n = [A.shape[0] for A in H.A]
    vec = 8 * (6 * n[0] + 6 * sum(n[1:]))  # r, z and the level buffers of one vector
    assert 40 * sum(n) < vec               # what is optional at load is less than that
    lo, hi = 0, 1 << 32
    while hi - lo > vec // 8:              # the least a load takes
        mid = (lo + hi) // 2
        S = Solver()
        S.set_alloc_limit(mid)
        try:
            S.load(H.A, H.P)
            hi = mid
        except AmgpsError as e:
            assert e.name == "AMGPS_E_NOMEM"
            lo = mid
        S.close()
    return hi + int(3.4 * vec)


@pytest.mark.parametrize("shape", [(13, 11, 9), (31, 26, 22)])
@pytest.mark.parametrize("coarse_kernel", [False, True])
def test_last_batch_of_one_vector(shape, coarse_kernel):
    import torch
    from paper_2407_09848_gb300.amgps import Solver
    H = _hierarchy(shape, 64)
    n = H.A[0].shape[0]
    limit = _limit_for_two(H)
    E = torch.from_numpy(pr.vec_normal(n, seed=1, count=5)).cuda()
    one, four = E.clone(), E[:4].clone()
    S = Solver().load(H.A, H.P)
    for i in range(5):
        S.error_cycles(one[i:i + 1], 2)
    S.close()
    S = Solver()
    S.set_alloc_limit(limit)
    S.load(H.A, H.P)
    S.set_coarse_kernel(coarse_kernel)
    S.vcycle(torch.from_numpy(pr.rhs_uniform(n, seed=3)).cuda(),
             torch.empty(n, dtype=torch.float64, device="cuda"))
    n4 = _launches(S, lambda: S.error_cycles(four, 2))  # 2 + 2
    n5 = _launches(S, lambda: S.error_cycles(E, 2))     # 2 + 2 + 1
    assert 2 * n5 == 3 * n4
    assert torch.equal(four, one[:4]) and torch.equal(E, one)
    S.close()


def test_more_vectors_than_blocks_in_y():
    import torch
    from paper_2407_09848_gb300.amgps import Solver
    H = _hierarchy((3, 3, 3), 8)
    S = Solver().load(H.A, H.P)
    m = 70000
    E = torch.from_numpy(pr.vec_normal(27, seed=1, count=m)).cuda()
    parts = E.clone()
    S.error_cycles(E, 1)
    for i in range(0, m, 30000):
        S.error_cycles(parts[i:i + 30000], 1)
    assert torch.equal(E, parts)
    S.close()
