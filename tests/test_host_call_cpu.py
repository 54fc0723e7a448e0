"""The native argument marshalling (csrc/host_call.cpp) against the one in Python, through a stand-in for the C entry point
that keeps a copy of the arguments it gets."""
import ctypes
import types

import numpy as np
import pytest
import torch

from paper_2506_18952_b200 import binding

lib = binding.load_library()
ENTRY = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.POINTER(binding.hola_verify_args), ctypes.c_void_p)


class _Ctx(binding.HolaVerify):
    def __init__(self, H, V):
        self.H, self.V, self.device, self._dev, self._ctx = H, V, 0, torch.device("cpu"), ctypes.c_void_p(16)
        self.lib = lib

    def close(self):
        pass


def _tensors(B, k, H, V, q=torch.bfloat16, w=torch.bfloat16, logits=False):
    W = torch.zeros(V, H, dtype=w)
    return dict(hidden=torch.zeros(B, k + 1, H, dtype=torch.bfloat16), W_lm=W, draft_tok=torch.zeros(B, k, dtype=torch.int32),
                draft_q=torch.zeros(B, k, V, dtype=q), uniforms=torch.zeros(B, k + 1),
                w_scale=torch.zeros(V) if w == torch.int8 else None), _Ctx(H, V).alloc_outputs(B, k, logits, device="cpu")


def _native(t, out, ctx, tau=1.5, draws=1, flags=0, gate=0, fallback=0, a8=False):
    got = []

    def entry(c, a, s):
        got.append((c, bytes(a.contents), s))
        return 7
    fn = ENTRY(entry)
    binding._entry["stand-in"] = ctypes.cast(fn, ctypes.c_void_p).value
    try:
        st = ctx._native("stand-in", t["hidden"], t["W_lm"], t["draft_tok"], t["draft_q"], t["uniforms"], tau, out, draws, flags,
                         gate, fallback, t["w_scale"], a8, types.SimpleNamespace(cuda_stream=32))
    finally:
        del binding._entry["stand-in"]
    if st is None:
        assert not got
        return None
    assert st == 7 and len(got) == 1 and got[0][0] == 16 and got[0][2] == 32
    return got[0][1]


def _python(t, out, ctx, tau=1.5, draws=1, flags=0, gate=0, fallback=0, a8=False):
    B, k1 = t["hidden"].shape[:2]
    a = ctx._args(t["hidden"], t["W_lm"], t["draft_tok"], t["draft_q"], t["uniforms"], tau, out, B, k1 - 1, gate, fallback,
                  t["w_scale"], a8, draws=bool(draws))
    a.flags = flags
    return bytes(a)


@pytest.mark.parametrize("k", [0, 3])
@pytest.mark.parametrize("q", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("w,a8", [(torch.bfloat16, False), (torch.int8, False), (torch.int8, True), (torch.int8, "a16")])
@pytest.mark.parametrize("gate,fallback,flags,tau,logits", [(0, 0, 0, 1.5, False), (1, 0, 1, float("inf"), True), (0, 1, 1, 2, True)])
def test_native_arguments_are_those_made_in_python(k, q, w, a8, gate, fallback, flags, tau, logits):
    t, out = _tensors(2, k, 64, 40, q, w, logits)
    ctx = _Ctx(64, 40)
    for draws in (1, 0):
        kw = dict(tau=tau, draws=draws, flags=flags, gate=gate, fallback=fallback, a8=a8)
        assert _native(t, out, ctx, **kw) == _python(t, out, ctx, **kw)
    t.update(draft_tok=None, draft_q=None, uniforms=None)
    kw = dict(tau=0.0, draws=0, flags=flags, a8=a8)
    assert _native(t, out, ctx, **kw) == _python(t, out, ctx, **kw)
    out.accept_len = out.logZ = out.status = None
    assert _native(t, out, ctx, a8=a8) == _python(t, out, ctx, a8=a8)
    t["W_lm"] = torch.nn.Parameter(t["W_lm"], requires_grad=False)
    assert _native(t, out, ctx, a8=a8) == _python(t, out, ctx, a8=a8)


class _Sub(torch.Tensor):
    pass


@pytest.mark.parametrize("change", [
    dict(hidden=torch.zeros(2, 4, 64)), dict(hidden=torch.zeros(2, 64, 4, dtype=torch.bfloat16).transpose(1, 2)),
    dict(hidden=torch.zeros(4, dtype=torch.bfloat16)), dict(hidden=None), dict(hidden=[1]), dict(W_lm=torch.zeros(40, 64)),
    dict(W_lm=torch.zeros(64, 40, dtype=torch.bfloat16).t()), dict(W_lm=object()), dict(w_scale=torch.zeros(40)),
    dict(W_lm=torch.zeros(40, 64, dtype=torch.int8)), dict(draft_q=torch.zeros(2, 3, 40, dtype=torch.float16)),
    dict(draft_tok=torch.zeros(3, 2, dtype=torch.int32).t()), dict(uniforms=torch.zeros(4, 2).t()),
    dict(uniforms=torch.zeros(2, 4).as_subclass(_Sub)), dict(tau="1"), dict(a8=True), dict(gate=1.0), dict(fallback=1 << 40),
    dict(out=object()), dict(hidden=torch.zeros(2, 4, 64, dtype=torch.bfloat16).to_sparse()),
])
def test_other_forms_are_left_to_python(change):
    t, out = _tensors(2, 3, 64, 40)
    assert _native(t, out, _Ctx(64, 40)) is not None
    out = change.pop("out", out)
    kw = {n: change.pop(n) for n in list(change) if n not in t}
    t.update(change)
    assert _native(t, out, _Ctx(64, 40), **kw) is None


@pytest.mark.parametrize("which", ["W8", "W4", "W16"])
def test_heads_of_mixed_widths(which):
    t, out = _tensors(2, 3, 128, 40)
    ctx = _Ctx(128, 40)
    buf = {"W16": torch.zeros(40, 128, dtype=torch.bfloat16), "W8": torch.zeros(40, 128, dtype=torch.int8),
           "W4": torch.zeros(40, 64, dtype=torch.uint8)}[which]
    bufs = {"W16": None, "W8": None, "W4": None, which: buf}
    head = binding.MixedHead(40, 128, [8], bufs["W16"], bufs["W8"], bufs["W4"], None, torch.zeros(40),
                             torch.zeros(1, dtype=torch.uint8), torch.zeros(1, dtype=torch.int32), binding.hola_wmix())
    t["W_lm"] = head
    for kw in (dict(), dict(gate=1, flags=1, tau=3.0), dict(draws=0)):
        assert _native(t, out, ctx, **kw) == _python(t, out, ctx, **kw)
    assert _native(t, out, ctx, a8=True) is None and _native(t, out, _Ctx(128, 41)) is None
    t["w_scale"] = torch.zeros(40)
    assert _native(t, out, ctx) is None
    t["w_scale"] = None
    setattr(head, which, torch.zeros(buf.shape[::-1], dtype=buf.dtype).t())
    assert _native(t, out, ctx) is None


class _Truth:
    """An object that has a truth value and nothing else."""

    def __init__(self, value):
        self.value = value

    def __bool__(self):
        return self.value


@pytest.mark.parametrize("wanted", [None, np.True_, np.bool_(False), torch.tensor(True), [], "yes", 2.5, _Truth(True)])
def test_outputs_take_the_truth_value_of_what_is_wanted(wanted):
    """Without a device the call ends where the first tensor is allocated: past the arguments."""
    def made(*flags):
        out = types.SimpleNamespace()
        try:
            binding._host.outputs(out, 0, 2, 4, 40, *flags)
        except RuntimeError:
            assert not torch.cuda.is_available()
            return None
        return out
    for out in (made(wanted, True, False), made(True, wanted, False), made(False, True, wanted)):
        assert out is None or out.entropy.shape == (2, 4)
    if torch.cuda.is_available():
        assert (made(wanted, False, False).logits is not None) == bool(wanted)
        assert hasattr(made(False, wanted, False), "next_tok") == hasattr(made(False, False, wanted), "draft_entropy") == bool(wanted)
    with pytest.raises(TypeError):
        binding._host.outputs(types.SimpleNamespace(), 0, "2", 4, 40, True, True, True)
    with pytest.raises(ValueError, match="ambiguous"):
        made(np.zeros(2), True, True)
