"""The launches that spread few rays over many warps, the step forms that the
FP32 march chooses by the lanes at work, and the system matrix from one trace:
every form gives the same bits, since a ray's arithmetic does not depend on
the lane, the warp's other rays or the kernel that runs it.
"""
import ctypes as C

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


@pytest.mark.parametrize("integrator", ["rk4", "heun"])
@pytest.mark.parametrize("n_tx", [2, 40, 128])
def test_path_matrix_from_one_trace(rt, n_tx, integrator, monkeypatch):
    prob = _problem(rt, n_tx)
    _, theta = _straight(prob)
    ds = 0.1 * prob.grid.h
    one = rt.rt_path_matrix(prob, theta, ds, integrator=integrator)
    monkeypatch.setattr(rt, "RECORD_BYTES", 0)     # count, count and fill
    three = rt.rt_path_matrix(prob, theta, ds, integrator=integrator)
    for a, b in zip(one, three):
        assert torch.equal(a, b)


def test_path_record_reports_rows_longer_than_its_capacity(rt):
    from paper_2511_18511_gb300 import _lib as L
    prob = _problem(rt, 24)
    _, theta = _straight(prob)
    ds = 0.1 * prob.grid.h
    want = rt.rt_path_matrix(prob, theta, ds)
    ctx = rt.default_context(prob.c.device.index)
    cap = 8                                        # most rows visit more cells
    runs = torch.empty(prob.n_pairs * cap * L.RUN_BYTES, dtype=torch.uint8, device="cuda")
    row_ptr = torch.full((prob.n_pairs + 1,), -1, dtype=torch.int64, device="cuda")
    nnz = C.c_int64(-1)
    ps, o, rec = prob.struct(), rt._opts(ds), L.RtRows(runs.data_ptr(), None, cap)
    s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = ctx.lib.rt_path_record(ctx.h, C.byref(ps), C.byref(o), C.c_void_p(theta.data_ptr()), C.byref(rec),
                                C.c_void_p(row_ptr.data_ptr()), C.byref(nnz), s)
    assert rc == L.RT_ENOMEM and nnz.value == want[1].numel()
    assert torch.equal(row_ptr, want[0])


def test_batch_of_several_is_each_alone(rt):
    """The instances' fans and adjoints run in one launch each; a batch of one
    gives the same bits, up to the order of the adjoint's FP64 sums (at most
    the 64 x 4 additions to a node here, 2^-53 of the sum of magnitudes each)."""
    probs = [_problem(rt, n, nx, ny, h) for n, nx, ny, h in ((33, 101, 96, 0.5), (2, 64, 70, 0.4), (70, 130, 128, 0.25))]

    def instances():
        out = []
        for p in probs:
            pairs, _ = _straight(p)
            d = (p.tx[pairs[:, 0].long()] - p.tx[pairs[:, 1].long()]).norm(dim=1)
            out.append(rt.BatchInstance.create(p, (d / 1.6).contiguous()))   # all weights of one sign: no cancellation
        return out

    batch = rt.rt_batch_run(instances(), 0.03, fan_ds=0.1)
    for b, alone in zip(batch, instances()):
        rt.rt_batch_run([alone], 0.03, fan_ds=0.1)
        for name in ("theta", "tof", "hit", "status", "iters"):
            assert torch.equal(getattr(b, name), getattr(alone, name))
        assert ((b.g_c - alone.g_c).abs() <= 1e-11 * alone.g_c.abs()).all()


# Nodes, frequencies and transducers at which the apply's items fill the SMs in
# chunks of 4 to 16 K-tiles, whole and ragged.
@pytest.mark.parametrize("n", [40, 97, 128])
@pytest.mark.parametrize("n_tx,n_freq", [(5, 1), (64, 8), (130, 3)])
def test_born_apply_chunks(rt, n, n_tx, n_freq):
    """The tensor-core product against the FP32 SIMT product of the same maps:
    both sum at most 12,900 nodes, whose FP32 roundings (2^-24 each, adding like
    a random walk) and the split's 2^-21 per product stay below 2e-5."""
    from paper_2511_18511_gb300 import phantoms as P
    h = 0.5
    R = 0.45 * n * h
    x = (torch.arange(n, dtype=torch.float64, device="cuda") - (n - 1) / 2) * h
    inside = x[None, :] ** 2 + x[:, None] ** 2 < R * R
    tx = torch.as_tensor(P.ring(n_tx, R), device="cuda")
    r = torch.sqrt((x[None, None, :] - tx[:, 0, None, None]) ** 2 + (x[None, :, None] - tx[:, 1, None, None]) ** 2)
    T = torch.where(inside, r / 1.5, torch.inf).float().contiguous()
    A = torch.where(inside, torch.rsqrt(r.clamp(min=h)), 0.0).float().contiguous()
    maps = rt.BornMaps(P.Grid(n, n, h), R, T, A)
    g = torch.Generator().manual_seed(n + n_tx)
    dc = torch.where(inside, torch.randn(n, n, generator=g, dtype=torch.float64).cuda(), 0.0).float().contiguous()
    f = [0.4 + 0.1 * k for k in range(n_freq)]
    a = rt.rtborn_apply(maps, f, dc, gemm="tf32x3").to(torch.complex128)
    b = rt.rtborn_apply(maps, f, dc, gemm="fp32").to(torch.complex128)
    assert float((a - b).abs().pow(2).sum().sqrt()) <= 2e-5 * float(b.abs().pow(2).sum().sqrt())
