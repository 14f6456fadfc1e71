"""The solve loop on the device after the context's state has changed, and at
tolerances whose square is not a normal number."""
import pytest

from paper_2407_09848_gb300 import problems as pr

pytestmark = pytest.mark.gpu


def _solver(shape, coarse_max=64):
    from paper_2407_09848_gb300.amgps import Solver
    H = pr.build_hierarchy(pr.varcoef(shape[0], 1.0, 4.0, seed=4, ny=shape[1], nz=shape[2]),
                           coarse_max)
    return Solver().load(H.A, H.P), H.A[0].shape[0]


def test_solve_after_the_coarse_kernel_was_switched_off():
    """The phases that the coarse kernel recorded for the old weights are not used again."""
    import torch
    out = []
    for recorded in (True, False):
        S, n = _solver((31, 26, 22))
        assert S.n_levels >= 3
        b = torch.from_numpy(pr.rhs_uniform(n, seed=1)).cuda()
        x, z = torch.empty_like(b), torch.empty_like(b)
        if recorded:
            S.set_coarse_kernel(True)
            S.vcycle(b, z)
            S.set_coarse_kernel(False)
        S.set_smoother(-1, "l1jacobi", 1)
        out.append((S.pcg(b, x, rtol=1e-8), x))
        S.close()
    assert out[0][0] == out[1][0] and torch.equal(out[0][1], out[1][1])


# squares: 1e-320 and 1e-324 are not normal (the latter rounds to 0), 1e-300 is
@pytest.mark.parametrize("rtol", [1e-150, 1e-160, 1e-162])
@pytest.mark.parametrize("outer", ["cg", "flexible", "fcg1"])
def test_tolerances_whose_square_underflows(rtol, outer):
    import torch
    S, n = _solver((19, 17, 13), 512)
    S.set_flexible(outer)
    b = torch.from_numpy(pr.rhs_uniform(n, seed=1) * 1e100).cuda()
    x, y = torch.empty_like(b), torch.empty_like(b)
    got = S.pcg(b, x, rtol=rtol, maxit=600, raise_on_noconv=False)
    S.profile(True)  # the host loop
    ref = S.pcg(b, y, rtol=rtol, maxit=600, raise_on_noconv=False)
    assert got == ref and torch.equal(x, y)
    S.close()
