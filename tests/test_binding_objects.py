"""The binding's objects as plain Python objects: what a program does with them besides passing them to the library.  No GPU."""
import copy
import gc
import io
import pickle
import weakref

import pytest
import torch

import paper_2502_20853_b200 as mx
from paper_2502_20853_b200 import build


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


def _filled(rows=96, cols=64, given=False):
    if given:
        q = mx.QMat(rows, cols, "cpu", torch.empty((rows, cols // 2), dtype=torch.uint8), torch.empty(mx.scale_bytes(rows, cols), dtype=torch.uint8))
    else:
        q = mx.QMat(rows, cols, "cpu")
    q.data.copy_(torch.arange(q.data.numel()).view(q.data.shape) % 251)
    q.scales.copy_(torch.arange(q.scales.numel()) % 241)
    return q


def _same(a, b):
    return type(a) is type(b) and (a.rows, a.cols) == (b.rows, b.cols) and torch.equal(a.data, b.data) and torch.equal(a.scales, b.scales)


@pytest.mark.parametrize("given", [False, True])
def test_matrix_is_copied_pickled_and_saved(given):
    q = _filled(given=given)
    q.note = "of layer 3"
    assert copy.copy(q).data.data_ptr() == q.data.data_ptr() and _same(copy.copy(q), q)
    for proto in range(pickle.HIGHEST_PROTOCOL + 1):
        assert _same(pickle.loads(pickle.dumps(q, proto)), q)
    f = io.BytesIO()
    osc = mx.OscState(torch.zeros(2, 2), q, torch.ones(2), torch.ones(3))
    torch.save(dict(osc=osc, ctx=mx.LinearCtx(q, q, seed=5)), f)
    f.seek(0)
    state = torch.load(f, weights_only=False)
    assert _same(state["osc"].wq_prev, q) and state["osc"].wq_prev.note == "of layer 3" and _same(state["ctx"].xq, q)
    for r in (copy.deepcopy(q), pickle.loads(pickle.dumps(q)), state["ctx"].wq):
        assert _same(r, q) and r.note == q.note and r.device == q.device
        r.data.zero_()
        r.scales.zero_()
        assert not _same(r, q) and q.data.any() and q.scales.any()
        assert (r.c().data, r.c().scales) == (r.data.data_ptr(), r.scales.data_ptr())


def test_matrix_saved_as_a_plain_object_is_loaded():
    """Objects pickled when the class was a plain one: its attributes are rows, cols, data and scales."""
    q = _filled()
    old = copy.copy(q)
    state = dict(rows=96, cols=64, data=q.data.clone(), scales=q.scales.clone())
    new = mx.QMat.__new__(mx.QMat)
    (new.__setstate__ if hasattr(new, "__setstate__") else new.__dict__.update)(state)
    assert _same(new, old) and new.c().data == state["data"].data_ptr() and new.device.type == "cpu"


def test_matrix_takes_other_tensors_and_attributes():
    q, other = _filled(), _filled(given=True)
    other.data.add_(1)
    q.data, q.scales = other.data, other.scales
    q.tag = 7
    assert _same(q, other) and q.tag == 7 and (q.c().data, q.c().scales) == (other.data.data_ptr(), other.scales.data_ptr())
    q.rows, q.cols = 48, 128
    assert (q.c().rows, q.c().cols) == (48, 128)
    w = weakref.ref(q)
    del q
    gc.collect()
    assert w() is None


def test_calls_follow_a_tensor_whose_storage_is_replaced():
    import ctypes as C
    seen = []
    entry = C.CFUNCTYPE(C.c_int32, C.c_void_p, C.c_int64, C.c_int64, C.c_int64, mx.binding.CMat, C.c_void_p, C.c_void_p, C.c_void_p)(
        lambda x, rows, cols, ld, dst, qp, status, stream: seen.append((dst.data, dst.scales)) or 0)
    address = C.cast(entry, C.c_void_p).value

    def call(q):
        assert mx.binding._host.quantize(address, None, q.rows, q.cols, q.cols, q, 0, 0, 0, 0, None, None) == 0
        return seen[-1]

    for q in (_filled(), _filled(given=True)):
        assert call(q) == (q.data.data_ptr(), q.scales.data_ptr())
        q.data.data = q.data.clone()            # e.g. moved elsewhere and back
        q.scales.set_(q.scales.clone())
        assert call(q) == (q.data.data_ptr(), q.scales.data_ptr()) == (q.c().data, q.c().scales) == (q.data_addr, q.scales_addr)
    q = mx.QMat(96, 64, "cpu")                  # nothing handed out yet
    assert call(q) == (q.data.data_ptr(), q.scales.data_ptr())


def test_c_structures_of_a_context_and_of_the_oscillation_state():
    xq, wq, xq_t, wq_t = (_filled() for _ in range(4))
    c = mx.LinearCtx(xq, wq, xq_t, -1, wq_t).c()
    assert [m.data for m in (c.xq, c.wq, c.xq_t, c.wq_t)] == [q.data.data_ptr() for q in (xq, wq, xq_t, wq_t)]
    assert c.xq_t_seed == c.wq_t_seed == 2 ** 64 - 1
    c = mx.LinearCtx(xq, wq).c()
    assert not c.xq_t.data and not c.wq_t.data and c.wq.rows == 96
    w, dw, dq = torch.zeros(3), torch.ones(3), torch.ones(4)
    c = mx.OscState(w, wq, dw, dq).c()
    assert (c.w_prev, c.wq_prev.scales, c.dist_w, c.dist_q) == (w.data_ptr(), wq.scales.data_ptr(), dw.data_ptr(), dq.data_ptr())


# every whole-number argument of every native call: None is no number
@pytest.mark.parametrize("name,numbers,pointers,matrices,n", [
    ("linear_fwd", (2, 3, 4, 6, 9, 14, 15), (1, 5, 7, 8, 16, 17, 18), (10, 11, 12, 13), 19),
    ("linear_bwd", (2, 9, 10, 11, 13, 15, 16, 19), (1, 12, 14, 17, 18, 20, 21), (3, 4, 5, 6, 7, 8), 22),
    ("quantize", (2, 3, 4, 6, 7, 8, 9), (1, 10, 11), (5,), 12),
    ("quantize_t", (3, 4, 5, 7, 8, 9, 10), (1, 11, 12), (2, 6), 13),
    ("qema_quantize", (4, 5, 6, 8), (1, 2, 9, 11, 12, 13, 14), (7, 10), 15)])
def test_native_calls_refuse_none_for_a_number(name, numbers, pointers, matrices, n):
    import ctypes as C
    called = []
    entry = C.CFUNCTYPE(C.c_int32)(lambda: called.append(1) or 0)
    fn, q = getattr(mx.binding._host, name), _filled()

    def call(**other):
        args = [0] * n
        args[0] = C.cast(entry, C.c_void_p).value
        for i in pointers:
            args[i] = None
        for i in matrices:
            args[i] = q
        if name == "qema_quantize":
            args[3] = 0.5
        for i, v in other.items():
            args[int(i[1:])] = v
        return fn(*args)

    assert call() == 0 and called
    for i in numbers:
        for bad in (None, 1.5, "1"):
            with pytest.raises(TypeError):
                call(**{"_%d" % i: bad})
    assert len(called) == 1


@pytest.mark.parametrize("rows,cols,shared", [(1024, 192, True), (2048, 768, False), (25216, 384, False)])
def test_matrices_of_a_call_share_memory_only_while_it_is_little(rows, cols, shared):
    """The two operands made from one tensor may be kept for different times: keeping one of them keeps no more than 1 MiB of the
    other's memory."""
    a, b = mx.QMat.two(rows, cols, cols, rows, "cpu")
    assert (a._buf is b._buf) == shared and a._buf.numel() <= (1 << 20 if shared else rows * cols)
    assert (a.rows, a.cols, b.rows, b.cols) == (rows, cols, cols, rows)
    assert a.data.shape == (rows, cols // 2) and b.scales.numel() >= mx.scale_bytes(cols, rows)


def test_stream_without_the_private_calls(monkeypatch):
    """A torch without the two internal functions: the public call gives the handle."""
    import importlib
    import types
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        monkeypatch.delattr(torch._C, name, raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=5))
    spec = importlib.util.spec_from_file_location("paper_2502_20853_b200._binding_again", mx.binding.__file__)
    again = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(again)
    assert again._stream() == 5
