"""rt_path_matrix where memory is short: the matrix from one trace keeps a
record of about the matrix's size, and a call that has room for the matrix
alone gives the same matrix by counting and filling."""
import ctypes as C
import types
import weakref

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
    from paper_2511_18511_gb300 import phantoms as P
    nx, h, n_tx = 101, 0.5, 96
    R = 0.42 * nx * h
    x = (np.arange(nx) - (nx - 1) / 2) * h
    c = 1500.0 * (1.0 + 0.03 * np.cos(x / 5.0)[None, :] * np.cos(x / 7.0)[:, None])
    prob = rt.Problem.create(P.Grid(nx, nx, h), c, P.ring(n_tx, R), R)
    e = torch.arange(n_tx, device="cuda").repeat_interleave(n_tx - 1)
    r = torch.arange(n_tx - 1, device="cuda").repeat(n_tx)
    d = prob.tx[r + (r >= e).long()] - prob.tx[e]
    theta = torch.atan2(d[:, 1], d[:, 0]).contiguous()
    ds = 0.1 * h
    return prob, theta, ds, rt.rt_path_matrix(prob, theta, ds)


class _Record:
    """torch.empty that notes the record's block and can refuse later ones."""

    def __init__(self, refuse=None):
        self.real, self.refuse, self.ref, self.size, self.stream = torch.empty, refuse, lambda: None, 0, None

    def __call__(self, *a, **k):
        if k.get("dtype") is self.refuse and self.ref() is not None:
            raise torch.OutOfMemoryError("no room beside the record")
        t = self.real(*a, **k)
        if k.get("dtype") is torch.uint8:
            self.ref, self.size, self.stream = weakref.ref(t), t.numel(), torch.cuda.current_stream()
        return t


class _Ctx:
    """A context whose library calls can be replaced."""

    def __init__(self, ctx, **calls):
        self.h, self.lib = ctx.h, type("Lib", (), {"__getattr__": lambda _, n: calls.get(n) or getattr(ctx.lib, n)})()


def _same(got, want):
    assert all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("refuse", [torch.int32, torch.float64])
def test_no_room_for_the_matrix_beside_the_record(rt, case, refuse, monkeypatch):
    prob, theta, ds, want = case
    empty = _Record(refuse)
    monkeypatch.setattr(torch, "empty", empty)
    _same(rt.rt_path_matrix(prob, theta, ds), want)
    assert empty.size > 0                          # the record was tried


def test_no_room_for_the_library_beside_the_record(rt, case, monkeypatch):
    """The record's block goes back to the device before the library is called again."""
    from paper_2511_18511_gb300 import _lib as L
    prob, theta, ds, want = case
    ctx = rt.default_context(prob.c.device.index)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.memory_reserved()
    empty = _Record()
    monkeypatch.setattr(torch, "empty", empty)
    reserved = []

    def matrix(*a):
        reserved.append(torch.cuda.memory_reserved())
        return ctx.lib.rt_path_matrix(*a)

    _same(rt.rt_path_matrix(prob, theta, ds, ctx=_Ctx(ctx, rt_path_record=lambda *a: L.RT_ENOMEM,
                                                      rt_path_matrix=matrix)), want)
    assert empty.size > 20 << 20 and empty.ref() is None
    assert reserved[0] < before + empty.size


def test_large_record_leaves_most_of_the_free_memory(rt, case, monkeypatch):
    from paper_2511_18511_gb300 import _lib as L
    prob, theta, ds, want = case
    ctx = rt.default_context(prob.c.device.index)
    calls = []

    def record(*a):
        calls.append(1)
        return ctx.lib.rt_path_record(*a)

    monkeypatch.setattr(rt, "RECORD_FREE_ASK", 0, raising=False)
    cap = ctx.lib.rt_rows_cap(prob.struct())
    size = prob.n_pairs * cap * L.RUN_BYTES
    for free, taken in ((4 * size, 1), (2 * size, 0)):
        # nothing of torch's cache counts here
        monkeypatch.setattr(torch.cuda, "mem_get_info", lambda dev=None: (free, 1 << 40))
        monkeypatch.setattr(torch.cuda, "memory_reserved", lambda dev=None: 0)
        monkeypatch.setattr(torch.cuda, "memory_allocated", lambda dev=None: 0)
        calls.clear()
        _same(rt.rt_path_matrix(prob, theta, ds, ctx=_Ctx(ctx, rt_path_record=record)), want)
        assert len(calls) == taken


@pytest.mark.parametrize("handle", [lambda s: s, lambda s: types.SimpleNamespace(cuda_stream=s.cuda_stream)])
def test_record_belongs_to_the_stream_that_uses_it(rt, case, handle, monkeypatch):
    """The allocator orders a block's uses on the stream it was taken on only."""
    prob, theta, ds, want = case
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    empty = _Record()
    monkeypatch.setattr(torch, "empty", empty)
    got = rt.rt_path_matrix(prob, theta, ds, stream=handle(side))
    assert empty.stream.cuda_stream == side.cuda_stream != torch.cuda.current_stream().cuda_stream
    side.synchronize()
    _same(got, want)


@pytest.mark.parametrize("cap", [1, 8, 31, 33])
@pytest.mark.parametrize("shift", [0, 1])
def test_rows_longer_than_their_record(rt, case, cap, shift):
    """Nothing is read past a row's record: the entries beyond it are column 0 and NaN."""
    from paper_2511_18511_gb300 import _lib as L
    prob, theta, ds, (row_ptr, col, val) = case
    ctx = rt.default_context(prob.c.device.index)
    runs = torch.empty(prob.n_pairs * cap * L.RUN_BYTES, dtype=torch.uint8, device="cuda")
    rp = torch.empty_like(row_ptr)
    nnz = C.c_int64(0)
    ps, o, rec = prob.struct(), rt._opts(ds), L.RtRows(runs.data_ptr(), None, cap)
    s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = ctx.lib.rt_path_record(ctx.h, C.byref(ps), C.byref(o), C.c_void_p(theta.data_ptr()), C.byref(rec),
                                C.c_void_p(rp.data_ptr()), C.byref(nnz), s)
    assert rc == L.RT_ENOMEM and nnz.value == col.numel() and torch.equal(rp, row_ptr)
    # shift 1: stores of single entries
    c = torch.full((shift + nnz.value,), -7, dtype=torch.int32, device="cuda")[shift:]
    v = torch.full((shift + nnz.value,), -7.0, dtype=torch.float64, device="cuda")[shift:]
    rc = ctx.lib.rt_path_expand(ctx.h, C.byref(ps), C.byref(rec), C.c_void_p(rp.data_ptr()), C.c_void_p(c.data_ptr()),
                                C.c_void_p(v.data_ptr()), s)
    assert rc == L.RT_OK
    row = torch.repeat_interleave(torch.arange(prob.n_pairs, device="cuda"), row_ptr.diff())
    kept = torch.arange(nnz.value, device="cuda") - row_ptr[row] < 4 * cap
    assert not bool(kept.all())
    assert torch.equal(c, torch.where(kept, col, 0))
    assert torch.equal(v[kept], val[kept]) and torch.isnan(v[~kept]).all()


def test_record_on_the_default_stream_by_its_handle(rt, case, monkeypatch):
    prob, theta, ds, want = case
    torch.cuda.synchronize()
    empty = _Record()
    monkeypatch.setattr(torch, "empty", empty)
    with torch.cuda.stream(torch.cuda.Stream()):
        got = rt.rt_path_matrix(prob, theta, ds, stream=types.SimpleNamespace(cuda_stream=0))
    assert empty.stream.cuda_stream == 0
    torch.cuda.synchronize()
    _same(got, want)
