"""Forms of the march that depend on how many rays a warp takes, in the kernels
that use them: one to three lanes (the FP32 step first tried inside the cell) and
more. A ray's result does not depend on it. And the FP64 march's reciprocal and
both forms of its renormalisation against the oracle's division and root."""
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


@pytest.fixture(scope="module")
def case(rt):
    """16,256 rays: 9 lanes a warp on 152 SMs in launches of 12 warps an SM."""
    from paper_2511_18511_gb300 import phantoms as P
    n, n_tx, h = 101, 128, 0.5
    R = 0.42 * n * h
    x = (np.arange(n) - (n - 1) / 2) * h
    c = 1500.0 * (1.0 + 0.04 * np.sin(x / 4.0)[None, :] * np.cos(x / 3.0)[:, None])
    prob = rt.Problem.create(P.Grid(n, n, h), c, P.ring(n_tx, R), R)
    e = torch.arange(n_tx, device="cuda").repeat_interleave(n_tx - 1)
    r = torch.arange(n_tx - 1, device="cuda").repeat(n_tx)
    r = r + (r >= e).long()
    d = prob.tx[r] - prob.tx[e]
    return prob, torch.stack([e, r], 1).to(torch.int32), torch.atan2(d[:, 1], d[:, 0]).contiguous()


def _subset(rt, case, n):
    """n rays spread over all, as a problem of its own: (selection, problem, angles)."""
    prob, pairs, theta = case
    sel = torch.arange(n, device="cuda") * pairs.shape[0] // n
    return sel, rt.Problem(prob.grid, prob.c, prob.tx, prob.ring_radius, pairs[sel].contiguous()), theta[sel].contiguous()


# 1,000, 2,500, 5,000 and 9,000 rays run on 1, 2, 3 and 5 lanes a warp.
@pytest.mark.parametrize("step", [0.1, 1.7])
@pytest.mark.parametrize("n", [1000, 2500, 5000, 9000])
def test_few_lanes_give_the_bits_of_many(rt, case, n, step):
    prob, _, theta = case
    ds = step * prob.grid.h
    sel, sub, th = _subset(rt, case, n)
    for a, b in zip(rt.rt_tof_forward(sub, th, ds), rt.rt_tof_forward(prob, theta, ds)):
        assert torch.equal(a, b[sel])
    row_ptr, col, val = rt.rt_path_matrix(prob, theta, ds)
    rp, c, v = rt.rt_path_matrix(sub, th, ds)
    length = row_ptr.diff()[sel]
    assert torch.equal(rp.diff(), length)
    at = torch.repeat_interleave(row_ptr[sel] - rp[:-1], length) + torch.arange(c.numel(), device="cuda")
    assert torch.equal(c, col[at]) and torch.equal(v, val[at])


@pytest.mark.parametrize("precision", ["fp32c", "fp64"])
def test_adjoint_on_few_lanes(rt, case, precision):
    """The adjoint of all rays is the sum of those of parts on 1 to 5 lanes: each
    ray adds the same numbers, in another order. A node takes 4 additions of each
    ray's visits at most; at 2^-53 of the largest sum each, 16,256 rays stay below
    1e-11 of it."""
    prob, pairs, theta = case
    ds = 0.1 * prob.grid.h
    w = 1.0 + 0.1 * torch.sin(torch.arange(pairs.shape[0], device="cuda", dtype=torch.float64))
    whole = rt.rt_tof_adjoint(prob, theta, w, ds, precision=precision)
    parts = torch.zeros_like(whole)
    order = torch.randperm(pairs.shape[0], generator=torch.Generator().manual_seed(5)).cuda()
    for sel in order.split([100, 1156, 2500, 4000, 8500]):
        sub = rt.Problem(prob.grid, prob.c, prob.tx, prob.ring_radius, pairs[sel].contiguous())
        parts += rt.rt_tof_adjoint(sub, theta[sel].contiguous(), w[sel].contiguous(), ds, precision=precision)
    assert float((parts - whole).abs().max()) <= 1e-11 * float(whole.abs().max())


@pytest.mark.parametrize("n", [1, 300, 3000])
def test_recording_link_on_few_lanes(rt, case, n):
    prob, _, _ = case
    ds = 0.1 * prob.grid.h
    sel, sub, _ = _subset(rt, case, n)
    whole = rt.rt_link_rows(prob, ds, rt.Rows.create(prob))
    rows = rt.Rows.create(sub)
    part = rt.rt_link_rows(sub, ds, rows)
    for name in ("theta", "tof", "hit", "status", "iters"):
        assert torch.equal(part[name], whole[name][sel])


@pytest.mark.parametrize("integrator,step", [("rk4", 0.5), ("rk4", 3.0), ("heun", 0.5), ("heun", 2.0)])
def test_fp64_step_in_a_steep_field(rt, orc, integrator, step):
    """Slopes of up to 0.2 a cell: |d|^2 leaves 1 by up to 7e-3 a step, so the
    renormalisation takes its series and its root. The roundings of the at most 100
    steps (a few 2^-53 each) act like a change of the launch angle of 1e-12 at most;
    T moves by 1e-3 of what a change of 1e-9 moves it, and its own sums round."""
    from paper_2511_18511_gb300 import phantoms as P
    n, n_tx = 61, 24
    x = np.arange(n) - (n - 1) / 2
    c = 1500.0 * (1.0 + 0.3 * np.sin(0.5 * x + 0.3)[None, :] * np.cos(0.55 * x)[:, None])
    R = 24.5
    g, tx = P.Grid(n, n, 1.0), P.ring(n_tx, R)
    prob = rt.Problem.create(g, c, tx, R)
    th = np.array([np.arctan2(*(tx[r] - tx[e])[::-1]) for e in range(n_tx) for r in range(n_tx) if r != e])
    with orc.integrator(integrator):
        want, move = (orc.tof(g, c, tx, R, step, th + q)[0] for q in (0.0, 1e-9))
    got = rt.rt_tof_forward(prob, torch.as_tensor(th, device="cuda"), step, precision="fp64", integrator=integrator)[0]
    assert (np.abs(got.cpu().numpy() - want) <= 1e-12 * want + 1e-3 * np.abs(move - want)).all()
