"""The per-iteration calls of the binding on the CPU: what Context hands to the library, and the extension module on its own."""
import ctypes as C
import gc
import subprocess
import sys
import weakref

import pytest
import torch

from paper_2502_20190_b200 import binding as b
from paper_2502_20190_b200 import build as tjbuild


class _Recorder:
    """Stands in for the extension module: every call is kept and succeeds."""

    def __init__(self):
        self.calls = []

    def __getattr__(self, name):
        def call(*args):
            self.calls.append((name, args))
            return (0, 1) if name == "publish_weights" else 0
        return call


@pytest.fixture(scope="module")
def lib():
    tjbuild.build()
    return b.load_library()


@pytest.fixture
def ctx(monkeypatch, lib):
    rec = _Recorder()
    monkeypatch.setattr(b, "_calls", rec)
    c = b.Context.__new__(b.Context)
    c.torch, c.device, c.h, c._addr, c._segments = torch, torch.device("cpu"), None, 4096, {}
    c._one, c.D, c.A, c.rec = torch.empty(1), 4, 2, rec
    return c


def _blobs(n, count):
    return [torch.zeros(n) for _ in range(count)]


def test_updates_hold_no_parameters(ctx):
    batch = dict(c=b.TjBatch())
    theta, target, m, v = _blobs(10, 4)
    refs = [weakref.ref(x) for x in (theta, target, m, v)]
    ctx.adam_step(batch, 1e-3, theta, target, m, v, 1)
    ctx.sgd_step(batch, 1e-3, theta, target)
    act = torch.zeros(3, dtype=torch.int32)
    ctx.ppo_step(torch.zeros(3, 4), act, *_blobs(3, 3), 1e-3, theta, m, v, 1)
    del theta, target, m, v
    gc.collect()
    assert [r() for r in refs] == [None] * 4


def test_updates_look_at_their_blobs_on_every_call(ctx):
    batch = dict(c=b.TjBatch())
    theta, target, m, v = _blobs(10, 4)
    ctx.adam_step(batch, 1e-3, theta, target, m, v, 1)
    target.resize_(4)                                 # the same tensor at the same address, smaller
    for call in (lambda: ctx.adam_step(batch, 1e-3, theta, target, m, v, 1), lambda: ctx.sgd_step(batch, 1e-3, theta, target)):
        with pytest.raises(AssertionError):
            call()
    wide = torch.zeros(10, 2)[:, 0]                   # right size, not contiguous
    with pytest.raises(AssertionError):
        ctx.sgd_step(batch, 1e-3, theta, wide)
    with pytest.raises(AssertionError):
        ctx.sgd_step(batch, 1e-3, theta, theta.double())


def test_numbers_are_taken_as_int_and_float_take_them(ctx):
    theta, target, m, v = _blobs(10, 4)
    ctx.adam_step(dict(c=b.TjBatch()), torch.tensor(0.5), theta, target, m, v, 3.0, beta1="0.5", eps=1)
    name, args = ctx.rec.calls[-1]
    assert name == "adam_step" and args[2:7] == (0.5, 0.5, 0.999, 1.0, 3) and all(type(a) is float for a in args[2:6]) and type(args[6]) is int
    act = torch.zeros(3, dtype=torch.int32)
    ctx.ppo_step(torch.zeros(3, 4), act, *_blobs(3, 3), 1, theta, m, v, torch.tensor(7))
    assert ctx.rec.calls[-1][1][7:15] == (1.0, 0.9, 0.999, 1e-8, 7, 0.2, 0.5, 0.01) and type(ctx.rec.calls[-1][1][11]) is int
    seg = dict(T=2, N=3, c=b.TjSegment())
    ctx.segment_minibatch(seg, torch.zeros(2, 3), torch.zeros(2, 3), 2.0, 4.0, dict(c=b.TjPpoMinibatch()))
    assert ctx.rec.calls[-1][1][4:6] == (2, 4) and all(type(a) is int for a in ctx.rec.calls[-1][1][4:6])
    ctx.sgd_step(dict(c=b.TjBatch()), 1, theta, target)
    assert ctx.rec.calls[-1][1][2] == 1.0


def test_a_status_outside_the_allowed_ones_raises(ctx):
    with pytest.raises(b.TjError):
        ctx._check(b.TJ_OK, (b.TJ_ERR_TIMEOUT,))
    assert ctx._check(b.TJ_ERR_TIMEOUT, (b.TJ_ERR_TIMEOUT,)) == b.TJ_ERR_TIMEOUT


def test_publish_takes_every_form_of_pointer(lib):
    host = (C.c_float * 3)()
    for blob in (None, 0, C.addressof(host), host, C.c_void_p(C.addressof(host)), C.pointer(host), b"blob"):
        for h in (None, C.c_void_p()):
            assert b.tj_publish_weights(h, blob, 12, 0) == (b.TJ_ERR_INVALID_ARG, 0)


def test_a_segment_comes_as_tensors_of_its_own(ctx, monkeypatch):
    ws = ctx.workspace = torch.zeros(4096, dtype=torch.uint8)
    seg, base = b.TjSegment(2, 3, 1), ws.data_ptr()
    seg.obs, seg.act, seg.rew, seg.done, seg.logp, seg.val = (base + 256 * i for i in range(6))
    monkeypatch.setattr(b, "tj_segment_acquire", lambda h: (b.TJ_OK, seg))
    first = ctx.segment_acquire()[1]
    first["obs"].requires_grad_()                      # what a caller does to its tensors stays with them
    first["rew"].unsqueeze_(0)
    second = ctx.segment_acquire()[1]
    assert not second["obs"].requires_grad and second["rew"].shape == (2, 3)
    assert all(second[k].data_ptr() == getattr(seg, k) for k in ("obs", "act", "rew", "done", "logp", "val"))


# arguments of each call with a null context; every one of them is refused by the library itself
NULL_CALLS = {
    "actor_step": (None, 1, None),
    "replay_sample": (None, -1, None, b.TjBatch()),
    "td_error": (None, b.TjBatch(), None, None, None),
    "publish_weights": (None, None, 12, 0),
    "sgd_step": (None, b.TjBatch(), 0.5, None, None, None),
    "adam_step": (None, b.TjBatch(), 0.5, 0.9, 0.99, 1e-8, 1, None, None, None, None, None),
    "ppo_step": (None, 3, None, None, None, None, None, 0.5, 0.9, 0.99, 1e-8, 1, 0.2, 0.5, 0.01, None, None, None, None),
    "gae": (None, None, None, None, 2, 3, 0.9, 0.9, None, None),
    "normalize": (None, None, 3, 1e-8, None),
    "segment_minibatch": (None, b.TjSegment(), None, None, 7, 0, b.TjPpoMinibatch()),
}
REFUSED = {name: (b.TJ_ERR_INVALID_ARG, 0) if name == "publish_weights" else b.TJ_ERR_INVALID_ARG for name in NULL_CALLS}


def test_the_library_loads_without_the_extension_module(lib, monkeypatch, tmp_path):
    monkeypatch.setattr(b, "_lib", None)
    monkeypatch.setattr(b, "_calls", None)
    monkeypatch.setattr(tjbuild, "CALLS", str(tmp_path / "_tjcall.none.so"))
    b.load_library()
    for name, args in NULL_CALLS.items():
        assert getattr(b._calls, name)(*args) == REFUSED[name], name


# ---- the extension module on its own
def test_module_refuses_calls_before_a_complete_init(lib):
    prog = """if True:
        import importlib.util, sys
        spec = importlib.util.spec_from_file_location("_tjcall", sys.argv[1])
        m = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(m)
        def raises(kind, f, *args):
            try:
                f(*args)
            except kind:
                return
            raise SystemExit("no " + kind.__name__)
        raises(RuntimeError, m.actor_step, None, 1, None)
        raises(ValueError, m.init, *[None] * 10)
        raises(TypeError, m.init, *[4096] * 9)
        raises(TypeError, m.init, *([4096] * 9 + ["x"]))
        raises(RuntimeError, m.gae, None, None, None, None, 1, 1, 0.5, 0.5, None, None)
    """
    r = subprocess.run([sys.executable, "-c", prog, tjbuild.CALLS], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)


@pytest.mark.parametrize("name", list(NULL_CALLS))
def test_module_arguments(lib, name):
    call, args = getattr(b._calls, name), list(NULL_CALLS[name])
    assert type(b._calls).__name__ == "module"
    assert call(*args) == REFUSED[name]                # a closed context: the library's own status, no crash
    for n in (0, len(args) - 1, len(args) + 1):
        with pytest.raises(TypeError, match="arguments"):
            call(*(args + [None])[:n])
    for i, a in enumerate(args):
        if isinstance(a, C.Structure):
            for other in (C.create_string_buffer(C.sizeof(a) + 1), C.c_int32(), 5, None):
                with pytest.raises(TypeError):
                    call(*args[:i], other, *args[i + 1:])
            continue
        for wrong in ("x", 1.5, object()):
            if isinstance(a, float) and wrong == 1.5:
                continue
            with pytest.raises(TypeError):             # nothing after the argument that failed is looked at
                call(*args[:i], wrong, *args[i + 1:])
        if isinstance(a, int):                         # integers are taken modulo 2^64 and narrowed, as by ctypes
            for big in (2 ** 63, 2 ** 70, -2 ** 65):
                assert call(*args[:i], big, *args[i + 1:]) == REFUSED[name]


class _Fails:
    def __init__(self, seen):
        self.seen = seen

    def __float__(self):
        self.seen.append("float")
        raise ZeroDivisionError("float")

    def __index__(self):
        self.seen.append("index")
        raise KeyError("index")


def test_module_passes_an_exception_on(lib):
    seen = []
    with pytest.raises(ZeroDivisionError):
        b._calls.sgd_step(None, b.TjBatch(), _Fails(seen), None, None, None)
    with pytest.raises(ZeroDivisionError):             # the first failure ends the call
        b._calls.adam_step(None, b.TjBatch(), 0.5, _Fails(seen), _Fails(seen), 1e-8, _Fails(seen), None, None, None, None, None)
    with pytest.raises(KeyError):
        b._calls.actor_step(None, _Fails(seen), None)
    assert seen == ["float", "float", "index"]
