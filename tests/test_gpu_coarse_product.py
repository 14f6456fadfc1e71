"""The coarsest level's product with the dense inverse at the edges of its
batches of columns (512, then 256 at a time), for one vector and for several."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc", [31, 512, 513, 767, 769, 1024])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_dense_solve(nc, prec):
    import torch
    from paper_2407_09848_gb300.amgps import Solver
    g = np.random.default_rng(nc)
    B = sp.random(nc, nc, 0.1, random_state=nc, format="csr")
    A = sp.csr_matrix(B + B.T)
    A = sp.csr_matrix(A + sp.diags(np.asarray(abs(A).sum(axis=1)).ravel() + 1.0))
    r = g.uniform(-1, 1, nc)
    ref = np.linalg.solve(A.toarray(), r)
    S = Solver().load([A], [], prec=prec)
    z = torch.empty(nc, dtype=torch.float64, device="cuda")
    S.vcycle(torch.from_numpy(r).cuda(), z)
    # FP32 hierarchies round r and z only
    tol = 1e-13 * nc if prec == "f64" else 1e-6
    assert np.linalg.norm(z.cpu().numpy() - ref) <= tol * np.linalg.norm(ref)
    S.close()


def test_several_vectors():
    """Error cycles of five vectors: the product takes four a warp."""
    import torch
    from paper_2407_09848_gb300 import problems as pr
    from paper_2407_09848_gb300.amgps import Solver
    H = pr.build_hierarchy(pr.poisson(19, 19, 19), 1024)
    assert 512 < H.A[-1].shape[0] <= 1024
    n = H.A[0].shape[0]
    S = Solver().load(H.A, H.P)
    E = torch.from_numpy(pr.vec_normal(n, seed=1, count=5)).cuda()
    one = E.clone()
    S.error_cycles(E, 2)
    for i in range(5):
        S.error_cycles(one[i:i + 1], 2)
    assert torch.equal(E, one)
    S.close()
