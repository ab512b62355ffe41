"""The launches that spread few rays over many warps and the step forms that the
FP32 march chooses by the lanes at work: every form gives the same bits, since
a ray's arithmetic does not depend on the lane or the warp's other rays.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2511_18511_gb300 as m
    return m


def _problem(rt, n_tx, nx=101, ny=96, h=0.5):
    from paper_2511_18511_gb300 import phantoms as P
    R = 0.42 * min(nx, ny) * h
    g = P.Grid(nx, ny, h)
    x = (np.arange(nx) - (nx - 1) / 2) * h
    y = (np.arange(ny) - (ny - 1) / 2) * h
    d2 = (x[None, :] - 0.2 * R) ** 2 + (y[:, None] + 0.3 * R) ** 2
    c = 1500.0 * (1.0 + 0.04 * np.exp(-d2 / (2 * (0.25 * R) ** 2)) + 0.01 * np.sin(x / 3.0)[None, :])
    return rt.Problem.create(g, c, P.ring(n_tx, R), R)


def _straight(prob):
    n = prob.n_tx
    e = torch.arange(n, device="cuda").repeat_interleave(n - 1)
    r = torch.arange(n - 1, device="cuda").repeat(n)
    r = r + (r >= e).long()
    d = prob.tx[r] - prob.tx[e]
    return torch.stack([e, r], 1).to(torch.int32), torch.atan2(d[:, 1], d[:, 0]).contiguous()


# 128 transducers: 16,256 rays, 7 lanes a warp on 152 SMs; the subsets run on
# one lane a warp (the sparse step form). Steps up to 1.7 cells cover samples
# beyond the neighbouring cell.
@pytest.mark.parametrize("integrator", ["rk4", "heun"])
@pytest.mark.parametrize("step", [0.1, 0.73, 1.7])
@pytest.mark.parametrize("precision,interpolator", [("fp32c", "bilinear"), ("fp64", "bilinear"), ("fp32c", "bspline")])
def test_forward_is_the_same_on_any_number_of_lanes(rt, precision, interpolator, step, integrator):
    prob = _problem(rt, 128)
    pairs, theta = _straight(prob)
    how = dict(precision=precision, interpolator=interpolator, integrator=integrator)
    ds = step * prob.grid.h
    t_all, hit_all = rt.rt_tof_forward(prob, theta, ds, **how)
    assert torch.isfinite(t_all).all()
    for n in (1, 31, 33, 700):
        sel = torch.arange(n, device="cuda") * (pairs.shape[0] // n)
        sub = rt.Problem(prob.grid, prob.c, prob.tx, prob.ring_radius, pairs[sel].contiguous())
        t, hit = rt.rt_tof_forward(sub, theta[sel].contiguous(), ds, **how)
        assert torch.equal(t, t_all[sel]) and torch.equal(hit, hit_all[sel])
