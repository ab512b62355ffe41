"""Stage points beyond the grid. The ring keeps one step and one cell from the
grid's edge, but a stage's direction is longer than 1 where the field is steep,
so with steps of several cells some stages sample outside. They take the edge
cell of each axis: a field whose outer three layers of nodes are equal gives the
same rays as that field continued by more such layers."""
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


# Of the rays that are compared 10 to 90 in a hundred sample outside in these cases
# (a march on the CPU); with samples of another row a quarter or more of those are
# off by more than 1e-4.
@pytest.mark.parametrize("precision", ["fp32c", "fp64"])
@pytest.mark.parametrize("field,rate,step,half,integrator", [("steep", 0.6, 6.0, 20, "rk4"), ("steep", 0.8, 4.0, 16, "heun"),
                                                             ("waves", 0.6, 6.0, 20, "rk4"),
                                                             ("waves", 0.6, 6.0, 20, "heun")])
def test_samples_outside_the_grid_take_the_edge_cell(rt, field, rate, step, half, integrator, precision):
    """The grids differ by whole cells and the transducers sit on multiples of
    2^-38, so the march's numbers are the same in each; the landing's FP64 sums
    differ in their last bits, which moves its FP32 step by a unit at most
    (2^-24): 1e-4 is far above that."""
    from paper_2511_18511_gb300 import phantoms as P
    n_tx = 64
    R = half - (step + 1) - 1 / 64
    x = np.arange(2 * half - 3) - (half - 2.0)
    if field == "steep":
        c = 1500 * np.exp(-rate * np.hypot(x[None, :] - 1.3, x[:, None] + 0.7))
    else:
        c = 1500 * (1 + 0.6 * np.sin(rate * x[None, :] + 0.3) * np.cos(1.1 * rate * x[:, None]))
    tx = np.round(P.ring(n_tx, R) * 2.0**38) / 2.0**38

    def T(layers):
        f = np.pad(c, layers, mode="edge")
        prob = rt.Problem.create(P.Grid(f.shape[1], f.shape[0], 1.0), f, tx, R)
        e = torch.arange(n_tx, device="cuda").repeat_interleave(n_tx - 1)
        r = torch.arange(n_tx - 1, device="cuda").repeat(n_tx)
        d = prob.tx[r + (r >= e).long()] - prob.tx[e]
        return rt.rt_tof_forward(prob, torch.atan2(d[:, 1], d[:, 0]).contiguous(), step, precision=precision,
                                 integrator=integrator)[0]

    got, more, want = T(2), T(34), T(130)
    inside = torch.isfinite(want) & (want != 0) & ((more / want - 1).abs() < 1e-5)   # rays that stay on the larger grids
    assert int(inside.sum()) > 500
    assert float((got / want - 1).abs()[inside].max()) < 1e-4
