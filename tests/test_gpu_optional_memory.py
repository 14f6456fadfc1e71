"""Arrays that only make a hierarchy faster (coarse corrections, the matrix of
the coarse sweeps) give way to what a later call needs, unless a graph that the
caller captured reads them."""
import numpy as np
import pytest

from paper_2407_09848_gb300 import problems as pr

pytestmark = pytest.mark.gpu


def _hierarchy(shape, coarse_max=512):
    return pr.build_hierarchy(pr.varcoef(shape[0], 1.0, 4.0, seed=2, ny=shape[1], nz=shape[2]),
                              coarse_max)


def _solver(H, limit=0, sweeps=0):
    from paper_2407_09848_gb300.amgps import Solver
    S = Solver()
    S.set_alloc_limit(limit)
    S.set_coarse_sweeps(sweeps)
    return S.load(H.A, H.P)


def _least(H):
    """Bytes of a load without anything optional (to 256)."""
    from paper_2407_09848_gb300.amgps import AmgpsError
    lo, hi = 0, 1 << 34
    while hi - lo > 256:
        mid = (lo + hi) // 2
        try:
            _solver(H, mid).close()
            hi = mid
        except AmgpsError as e:
            assert e.name == "AMGPS_E_NOMEM"
            lo = mid
    return hi


def _reverse_bytes(H):
    """The reverse-mode buffers: six vectors a level (two on the coarsest), the sums of a loss."""
    n = [A.shape[0] for A in H.A]
    return 8 * (6 * sum(n[:-1]) + 2 * n[-1]) + 8 * (32 * 32 + 2 * 4096) + 4096


@pytest.mark.parametrize("sweeps", [0, 30])
@pytest.mark.parametrize("call", ["loss", "smooth", "vcycle"])
def test_reverse_mode_fits_where_the_load_and_its_buffers_do(call, sweeps):
    import torch
    H = _hierarchy((31, 26, 22))
    n = H.A[0].shape[0]
    limit = _least(H) + _reverse_bytes(H)
    r, g = (torch.from_numpy(pr.rhs_uniform(n, seed=i)).cuda() for i in (1, 2))
    E = torch.from_numpy(pr.vec_normal(n, seed=1, count=3)).cuda()
    z = torch.empty_like(r)

    def run(S):
        S.vcycle(r, z)  # builds the graphs, with whatever is optional
        if call == "loss":
            out = S.loss_grad(E)
        elif call == "smooth":
            gb, gx, gw = S.smooth_backward(0, "cheb4_opt", 4, r, None, g)
            out = (gb.cpu().numpy(), gw)
        else:
            gr, gw = S.vcycle_backward(r, g)
            out = (gr.cpu().numpy(), gw)
        S.vcycle(r, z)
        x = torch.empty_like(r)
        it = S.pcg(r, x)[0]
        S.close()
        return [np.asarray(o) for o in out] + [z.cpu().numpy(), x.cpu().numpy(), it]
    lim, free = run(_solver(H, limit, sweeps)), run(_solver(H, 0, sweeps))
    assert lim[-1] == free[-1]
    for a, b in zip(lim[:-1], free[:-1]):
        # the correction in another form, sums over vectors in another order
        assert np.linalg.norm(a - b) <= 1e-11 * np.linalg.norm(b)


def test_corrections_stay_when_they_would_not_make_enough_room():
    """Operators of degree 8 do not fit even without the corrections: those are kept."""
    import torch
    H = _hierarchy((57, 51, 48))
    n = H.A[0].shape[0]
    r = torch.from_numpy(pr.rhs_uniform(n, seed=1)).cuda()
    z = [torch.empty_like(r) for _ in range(2)]
    S = _solver(H)
    S.vcycle(r, z[0])
    S.set_alloc_limit(1)
    S.set_smoother(0, "cheb4_opt", 8)
    S.set_smoother(0, "cheb4_opt", 4)
    S.vcycle(r, z[1])
    assert torch.equal(z[0], z[1])
    S.close()


def test_corrections_come_back_with_a_smaller_degree():
    import torch
    H = _hierarchy((57, 51, 48))
    n = H.A[0].shape[0]
    r = torch.from_numpy(pr.rhs_uniform(n, seed=1)).cuda()
    z = [torch.empty_like(r) for _ in range(3)]
    S = _solver(H)
    stored = S.level_info(0)[2]
    S.set_smoother(0, "cheb4_opt", 2)
    S.vcycle(r, z[0])
    S.close()
    # three operators at load (degree 4) and the corrections (36 B a row); one more
    # operator (56 B a row) fits only without level 0's correction
    S = _solver(H, _least(H) + 3 * 8 * stored + 60 * n)
    S.set_smoother(0, "cheb4_opt", 5)
    S.vcycle(r, z[1])
    S.set_smoother(0, "cheb4_opt", 2)
    S.vcycle(r, z[2])
    assert torch.equal(z[0], z[2]) and not torch.equal(z[0], z[1])
    S.close()


@pytest.mark.parametrize("what", ["operators", "reverse", "sweeps"])
def test_a_captured_cycle_keeps_its_arrays(what):
    """The caller's graph gives the same bits after a call that would like their place."""
    import torch
    from paper_2407_09848_gb300.amgps import AmgpsError, Solver
    H = _hierarchy((57, 51, 48))
    n = H.A[0].shape[0]
    least = _least(H)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        r = torch.from_numpy(pr.rhs_uniform(n, seed=1)).cuda()
        z = torch.empty_like(r)
        S = Solver(stream=s.cuda_stream)
        S.set_step_form(0)
        S.set_coarse_sweeps(30 if what == "sweeps" else 0)
        S.load(H.A, H.P)
        S.vcycle(r, z)
        s.synchronize()
        ref = z.clone()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            S.vcycle(r, z)
        if what == "operators":      # three would fit without the corrections
            S.set_alloc_limit(least + 3 * 8 * S.level_info(0)[2] + 4096)
            S.set_step_form(1)
        elif what == "reverse":
            S.set_alloc_limit(least + _reverse_bytes(H))
            with pytest.raises(AmgpsError, match="AMGPS_E_NOMEM"):
                S.smooth_backward(0, "cheb4_opt", 4, r, None, ref)
        else:
            S.set_coarse_sweeps(7)
        z.zero_()
        g.replay()
        s.synchronize()
        assert torch.equal(z, ref)
    S.close()
