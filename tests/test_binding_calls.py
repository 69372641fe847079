"""The calls marshalled in C (csrc/wpp_call.c) refuse on the host what the ctypes calls refuse: no GPU is touched, the context
is null throughout and the library itself answers WPP_ERR_INVALID_ARG to what passes."""
import ctypes
import sys

import pytest
import torch

import paper_2609_35263_b200.binding as B


class _NoContext:
    handle, device = ctypes.c_void_p(), 0


class _Stream:
    cuda_stream = 0


class _Plan:
    def __init__(self, host, dev=None):
        self.host, self.dev = host, dev


CTX, PLAN, T = _NoContext(), _Plan(torch.zeros(256, dtype=torch.uint8)), torch.zeros(4)
DESC = B.make_desc(1, 2, 1, 128, 16, 4, 8)


def _append(desc=DESC, plan=PLAN, ctx=CTX, **kw):
    B.load_library()
    a = dict(k_new=T, v_new=T, k_cache=T, v_cache=T, block_tables=T, prefix_lens=T, chunk_lens=T)
    status = kw.pop("status", None)
    a.update(kw)
    B.wpp_kv_append(ctx, desc, *a.values(), plan, status=status, stream=_Stream())


def _attention(desc=DESC, plan=PLAN, ctx=CTX, **kw):
    B.load_library()
    a = dict(q=T, out=T, lse=None, k_cache=T, v_cache=T, block_tables=T, prefix_lens=T, chunk_lens=T)
    more = {k: kw.pop(k) for k in ("workspace", "status") if k in kw}
    a.update(kw)
    B.wpp_prefill_attention_varlen(ctx, desc, *a.values(), plan, stream=_Stream(), **more)


def _kda(ctx=CTX, **kw):
    B.load_library()
    x, i = torch.zeros(4, 1, 128), torch.zeros(2, dtype=torch.int64)
    a = dict(q=x, k=x, v=x, alpha=x, beta=x, row_offsets=i, state_pool=torch.zeros(1, 1, 128, 128), state_in=T, state_out=T, out=x,
             stream=_Stream())
    a.update(kw)
    B.wpp_kda_chunk(ctx, **a)


@pytest.mark.parametrize("call", [_append, _attention, _kda])
def test_a_null_context_reaches_the_library(call):
    with pytest.raises(B.WppError) as e:
        call()
    assert e.value.status == 1
    with pytest.raises(B.WppError):
        call(status=torch.zeros(1, dtype=torch.int32))


@pytest.mark.parametrize("value", [0, 1, False, True, 2 ** 40, "x"])
@pytest.mark.parametrize("call,names", [
    (_append, ["k_new", "v_new", "k_cache", "v_cache", "block_tables", "prefix_lens", "chunk_lens", "status"]),
    (_attention, ["q", "out", "lse", "k_cache", "v_cache", "block_tables", "prefix_lens", "chunk_lens", "workspace", "status"]),
    (_kda, ["k", "alpha", "beta", "state_in", "state_out", "prefix_lens", "out", "workspace", "status"]),
])
def test_an_integer_is_no_memory(call, names, value):
    for name in names:
        with pytest.raises(AttributeError):
            call(**{name: value})


@pytest.mark.parametrize("call", [_append, _attention])
@pytest.mark.parametrize("host,dev", [(None, None), (T.data_ptr(), None), (T, 0), (T, 64)],
                         ids=["no host buffer", "integer host", "dev 0", "dev 64"])
def test_a_plan_has_a_host_buffer_and_no_integers(call, host, dev):
    with pytest.raises(AttributeError):
        call(plan=_Plan(host, dev))


@pytest.mark.parametrize("call", [_append, _attention])
@pytest.mark.parametrize("desc", [bytes(ctypes.sizeof(B.BatchDesc)), bytearray(ctypes.sizeof(B.BatchDesc)), B.KdaDesc(), None, 0,
                                  ctypes.byref(DESC), (ctypes.c_char * ctypes.sizeof(B.BatchDesc))()],
                         ids=["bytes", "bytearray", "other", "none", "integer", "byref", "array"])
def test_a_description_is_one(call, desc):
    with pytest.raises(TypeError):
        call(desc=desc)


def test_what_derives_from_a_description_is_one():
    class Mine(B.BatchDesc):
        _fields_ = [("own", ctypes.c_int64)]

    with pytest.raises(B.WppError):
        _append(desc=Mine())


class _Pointer:
    def __init__(self, value):
        self.value = value

    def data_ptr(self):
        if isinstance(self.value, Exception):
            raise self.value
        return self.value


@pytest.mark.parametrize("value,error", [("0", TypeError), (None, TypeError), (1.0, TypeError), (2 ** 80, OverflowError),
                                         (KeyError("mine"), KeyError)])
def test_an_address_is_an_integer_of_the_machine(value, error):
    with pytest.raises(error):
        _append(k_new=_Pointer(value))


def test_a_missing_module_is_answered_with_the_build_instruction(monkeypatch):
    B.load_library()
    name = B.__package__ + "._wpp_call"
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.delattr(sys.modules[B.__package__], "_wpp_call", raising=False)
    monkeypatch.setitem(sys.modules, name, None)                        # what a failed search leaves
    with pytest.raises(ImportError, match="python -m paper_2609_35263_b200.build"):
        B.load_library()
    assert B._lib is None


def test_the_compiler_is_looked_for(monkeypatch, tmp_path):
    from paper_2609_35263_b200 import build
    mine = tmp_path / "mine"
    mine.write_text("#!/bin/sh\n")
    mine.chmod(0o755)
    monkeypatch.setenv("CC", str(mine))
    assert build._cc() == [str(mine)]
    monkeypatch.setenv("CC", str(mine) + " -m64")
    assert build._cc() == [str(mine), "-m64"]
    monkeypatch.setenv("CC", "")
    monkeypatch.setenv("PATH", str(tmp_path))
    with pytest.raises(RuntimeError, match="C compiler"):
        build._cc()
