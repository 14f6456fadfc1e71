"""The solve loop on the device against the host loop (which a solve takes while
its kernels are being timed): same bits, counts and residuals, same errors."""
import numpy as np
import pytest

from paper_2407_09848_gb300 import problems as pr

pytestmark = pytest.mark.gpu


def _solver(shape, prec, outer):
    from paper_2407_09848_gb300.amgps import Solver
    H = pr.build_hierarchy(pr.varcoef(shape[0], 1.0, 4.0, seed=4, ny=shape[1], nz=shape[2]), 512)
    S = Solver().load(H.A, H.P, prec=prec)
    S.set_flexible(outer)
    return S, H.A[0].shape[0]


# one level (dense solve only), a few small levels, and a level 0 in the
# stored-operator form (c = M^-1 r fused into the r update)
@pytest.mark.parametrize("shape", [(7, 6, 5), (19, 17, 13), (61, 48, 46)])
@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("outer", ["cg", "flexible", "fcg1"])
def test_device_loop_equals_host_loop(shape, prec, outer):
    import torch
    S, n = _solver(shape, prec, outer)
    x, y = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    for seed in (1, 2):  # the second solve runs the graph again on other vectors
        b = torch.from_numpy(pr.rhs_uniform(n, seed=seed)).cuda()
        S.profile(False)
        got = S.pcg(b, x, rtol=1e-8)
        S.profile(True)
        ref = S.pcg(b, y, rtol=1e-8)
        assert got == ref and torch.equal(x, y)
        S.profile(False)
        # stopped by maxit: the last iterate
        got = S.pcg(b, x, rtol=1e-14, maxit=3, raise_on_noconv=False)
        S.profile(True)
        ref = S.pcg(b, y, rtol=1e-14, maxit=3, raise_on_noconv=False)
        assert got == ref and torch.equal(x, y)
    S.close()


@pytest.mark.parametrize("outer", ["cg", "flexible", "fcg1"])
def test_device_loop_zero_and_not_finite(outer):
    import torch
    from paper_2407_09848_gb300.amgps import AmgpsError
    S, n = _solver((19, 17, 13), "f64", outer)
    b = torch.zeros(n, dtype=torch.float64, device="cuda")
    x = torch.ones_like(b)
    assert S.pcg(b, x) == (0, 0.0) and not x.any()
    b[5] = float("nan")
    with pytest.raises(AmgpsError) as e:
        S.pcg(b, x)
    assert e.value.name == "AMGPS_E_NAN"
    b[5] = 1.0                      # the context stays usable
    it, rel = S.pcg(b, x, rtol=1e-8)
    assert it > 0 and rel <= 1e-8
    # new weights rebuild the loop
    S.set_smoother(-1, "cheb1_opt", 2)
    it2, rel2 = S.pcg(b, x, rtol=1e-8)
    assert rel2 <= 1e-8
    S.close()
