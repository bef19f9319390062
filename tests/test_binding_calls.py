"""The argument-converting extension and its ctypes stand-in convert alike: both reach the library's argument checks
with what the caller gave (no GPU: the calls are rejected, or return before anything is launched)."""
import ctypes as C

import numpy as np
import pytest


@pytest.fixture(scope="module")
def calls():
    from paper_2411_18462_b200 import binding, build
    build.build()
    lib = binding.library()
    assert type(binding._calls).__name__ == "module", "the extension was not built"
    return binding._calls, binding._CtypesCalls(lib)


class Tensor:
    def data_ptr(self):
        return 1 << 20


class Stream:
    cuda_stream = 0


def draft(f, handle, **over):
    a = dict(logits=Tensor(), dtype=0, B=0, V=8, stride=8, T=1.0, thresh=0.3, uniforms=Tensor(), token=1 << 20,
             entropy=Tensor(), stop=Tensor(), stats=None, stream=Stream())
    a.update(over)
    return f(handle, *a.values())


def test_both_give_the_same_status(calls):
    ctx = C.create_string_buffer(4096)          # never looked into: an empty batch returns before that
    h = C.addressof(ctx)
    cases = [({}, 0), (dict(B=np.int32(0), V=np.int64(8)), 0), (dict(T=np.float32(1.0), thresh=1), 0), (dict(T=0, uniforms=None), 0),
             (dict(T=-1.0), -1), (dict(T=float("inf")), -1), (dict(thresh=float("nan")), -1), (dict(dtype=7), -2), (dict(V=0), -1),
             (dict(logits=None), -1), (dict(uniforms=None), -1), (dict(logits=(1 << 20) + 1), -1), (dict(stream=0), 0),
             (dict(stream=None), 0), (dict(B=-1), -1)]
    for over, want in cases:
        for c in calls:
            assert draft(c.draft_step, h, **over) == want, (over, c)
    for c in calls:
        assert draft(c.draft_step, 0) == -1
        assert c.graph_launch(0, Stream()) == -1


def test_bad_arguments_raise(calls):
    for c in calls:
        with pytest.raises(TypeError):
            c.draft_step(0, 1, 2)
        with pytest.raises(AttributeError):
            draft(c.draft_step, 0, logits=object())
        with pytest.raises((TypeError, ValueError)):
            draft(c.draft_step, 0, T="warm")


def test_what_the_conversions_take_and_refuse(calls):
    from paper_2411_18462_b200 import binding
    for c in calls:
        assert draft(c.draft_step, C.addressof(C.create_string_buffer(4096)), T="1.0", B=0.0) == 0    # as float() and int() do
    ctx = object.__new__(binding.Context)
    ctx._h, ctx._hv = C.c_void_p(), 0
    args = dict(logits=Tensor(), dtype=0, B=0, V=8, stride=8, T=1.0, thresh=0.3, uniforms=Tensor(), token=1 << 20, entropy=Tensor(),
                stop=Tensor(), stats=None, stream=Stream())
    with pytest.raises(binding.SvipError):
        ctx.bind("draft_step", *args.values())()           # no context: the library refuses it
    for over in (dict(B=2.5), dict(V="8"), dict(T="1.0"), dict(dtype=None)):
        with pytest.raises(TypeError):
            ctx.bind("draft_step", *dict(args, **over).values())
