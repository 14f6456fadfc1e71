"""Stored-operator steps through the TMA-fed kernel (asked for: these grids are
below its default size) against the direct kernel: same bits, one smoother and
one V-cycle, FP64; and the FP32 and BF16 recurrence steps the same way."""
import pytest

from paper_2407_09848_gb300 import problems as pr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(72, 72, 64), (57, 53, 47)])
@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("kind,k", [("cheb4_opt", 4), ("cheb4_opt", 6), ("cheb1_opt", 3), ("l1jacobi", 2)])
def test_tma_equals_direct(shape, prec, kind, k):
    import torch
    from paper_2407_09848_gb300.amgps import Solver
    H = pr.build_hierarchy(pr.varcoef(shape[0], 1.0, 4.0, seed=2, ny=shape[1], nz=shape[2]), 512)
    S = Solver().load(H.A, H.P, prec=prec)
    S.set_smoother(-1, kind, k)
    n = H.A[0].shape[0]
    b, x0 = (torch.from_numpy(pr.rhs_uniform(n, seed=i)).cuda() for i in (1, 2))
    out = []
    for tma in ("always", False):
        S.set_tma(tma)
        x, z = x0.clone(), torch.empty_like(b)
        S.smooth(0, kind, k, b, x, x_is_zero=False)
        S.vcycle(b, z)
        out.append((x, z))
    S.synchronize()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    S.close()
