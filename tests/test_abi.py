"""The C-ABI library loads without a GPU, exports every declared symbol, and rejects bad arguments
before touching the device."""
import ctypes
import importlib.util
import os
import re
import sys

import pytest
import torch

from paper_2306_15799_b200 import binding, build
from paper_2306_15799_b200.configs import PERFORMER, RNN

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load()


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "flurka.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(flurka_[a-z_0-9]+)\s*\(", text)))


def test_exports_every_declared_symbol(lib):
    names = _declared_symbols()
    assert "flurka_forward" in names and "flurka_forward_host" in names and len(names) >= 12
    for n in names:
        assert hasattr(lib, n), "libflurka.so does not export %s" % n
    assert sorted(binding.EXPORTS) == [n for n in names if n in binding.EXPORTS]
    assert set(binding.EXPORTS) <= set(names)
    assert lib.flurka_version() == 100


def test_strerror_is_static_text(lib):
    for code in range(-9, 1):
        s = lib.flurka_strerror(code)
        assert isinstance(s, bytes) and len(s) > 1
    assert b"NULL" in lib.flurka_strerror(-1)


def test_argument_checks_need_no_device(lib):
    buf = ctypes.create_string_buffer(1 << 16)
    base = (ctypes.addressof(buf) + 255) & ~255
    q, k, v, e, f, w, o = (base + 4096 * i for i in range(7))
    fwd = lib.flurka_forward
    ok = dict(variant=0, B=1, H=1, N=8, d=8, k=4, m=8)

    def call(Q=q, K=k, V=v, E=e, F=f, W=w, out=o, **kw):
        a = dict(ok); a.update(kw)
        return fwd(Q, K, V, E, F, W, a["variant"], a["B"], a["H"], a["N"], a["d"], a["k"], a["m"], out, None)

    assert call(Q=None) == -1 and call(out=None) == -1 and call(W=None) == -1
    assert call(W=None, variant=1) in (-7, 0)          # RNN needs no W; only the device is missing
    assert call(variant=7) == -2 and call(variant=0x800) == -2
    assert call(variant=0x200) in (-7, 0)              # [B,N,H,d] layout flag is valid
    assert call(N=0) == -3 and call(d=129) == -3 and call(k=0) == -3 and call(m=0) == -3 and call(k=5000) == -3
    assert call(B=70000) == -3
    assert call(Q=q + 2) == -4 and call(out=o + 8) == -4
    assert call(out=q) == -8 and call(out=e) == -8
    import torch
    if not torch.cuda.is_available():
        assert call() == -7                              # valid arguments, but no sm_100 device
    assert lib.flurka_workspace_bytes(0, 1, 2, 256, 32, 32, 64) > 2 * 2 * 32 * 32 * 4
    assert lib.flurka_workspace_bytes(9, 1, 2, 256, 32, 32, 64) == 0
    assert lib.flurka_set_workspace(ctypes.c_void_p(base + 8), 1024) == -4
    assert lib.flurka_set_workspace(None, 0) == 0
    prev = lib.flurka_set_path(1)
    assert lib.flurka_set_path(prev) == 1
    assert lib.flurka_debug_copy(0, ctypes.c_void_p(base), 16, None) == -5   # no forward has run yet


def test_binding_rejects_bad_tensors():
    import torch
    from paper_2306_15799_b200 import PERFORMER
    Q = torch.zeros(1, 1, 8, 8)
    E = torch.zeros(4, 8)
    W = torch.zeros(8, 8)
    with pytest.raises(ValueError):
        binding.flurka_forward(Q, Q, Q, E, E, W, PERFORMER)          # CPU tensors on the device entry
    with pytest.raises(ValueError):
        binding.flurka_forward_host(Q, Q, Q, torch.zeros(4, 9), E, W, PERFORMER, out=torch.zeros_like(Q))
    with pytest.raises(TypeError):
        binding.flurka_forward_host(Q.half(), Q.half(), Q.half(), E.half(), E.half(), W.half(), PERFORMER,
                                    out=torch.zeros_like(Q).half())


@pytest.fixture(scope="module")
def cpu_marshal(tmp_path_factory):
    """csrc/marshal.cpp for tensors on the CPU, in front of functions that record what they are given: (module, calls)."""
    text = open(build.MARSHAL_SOURCE).read()
    for old, new in (("t.is_cuda()", "t.is_cpu()"), ("c10::cuda::getCurrentCUDAStream().stream()", "nullptr")):
        assert text.count(old) == 1
        text = text.replace(old, new)
    folder = tmp_path_factory.mktemp("marshal")
    source, target = str(folder / "marshal.cpp"), str(folder / "_marshal.so")
    open(source, "w").write(text)
    build.compile_marshal(source, target)
    spec = importlib.util.spec_from_file_location("_marshal", target)
    module = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(module)
    calls = []
    vp, ci = ctypes.c_void_p, ctypes.c_int
    record = lambda *a: calls.append(a) or 0
    forward = ctypes.CFUNCTYPE(ci, *[vp] * 6, *[ci] * 7, vp, vp)(record)
    backward = ctypes.CFUNCTYPE(ci, *[vp] * 7, *[ci] * 7, *[vp] * 6)(record)
    module.init(ctypes.cast(forward, vp).value, ctypes.cast(backward, vp).value)
    yield module, calls
    del forward, backward


def _small_call(layout="bhnd", per_head=False, dtype=torch.float32):
    B, H, N, d, k, m = 2, 3, 12, 8, 5, 7
    shape = (B, N, H, d) if layout == "bnhd" else (B, H, N, d)
    r = lambda *s: torch.randn(*s).to(dtype)
    ef = (H, k, N) if per_head else (k, N)
    return (B, H, N, d, k, m), [r(*shape), r(*shape), r(*shape), r(*ef), r(*ef), r(m, d)], r(*shape)


@pytest.mark.parametrize("transform", ["vmap", "grad", "jvp", "grad of others"])
def test_tensors_without_memory_are_left_to_the_python_path(cpu_marshal, transform):
    """Inside torch.func's transforms a tensor has a type, a device and strides but no memory: the module declines such a
    call (binding.py then raises RuntimeError) with the interpreter in hand."""
    module, calls = cpu_marshal
    _, (Q, *rest), dO = _small_call()
    seen = []

    def call(q):
        del calls[:]
        seen.append(module.forward(q, *rest, PERFORMER, False))
        seen.append(module.backward(q, *rest, PERFORMER, False, dO))
        seen.append(module.backward(Q, *rest, PERFORMER, False, q))
        assert not calls
        with pytest.raises(RuntimeError):
            q.data_ptr()
        return q.sum()

    def others(q):                             # (what is allocated inside has no memory either)
        del calls[:]
        seen.append(module.forward(Q, *rest, PERFORMER, False))
        assert not calls
        return q.sum()

    if transform == "vmap":
        torch.func.vmap(call)(torch.stack([Q, Q]))
    elif transform == "grad":
        torch.func.grad(call)(Q)
    elif transform == "jvp":
        torch.func.jvp(call, (Q,), (torch.ones_like(Q),))
    else:
        torch.func.grad(others)(Q.clone())
    assert seen and all(s is None for s in seen)


class _Subclass(torch.Tensor):
    pass


@pytest.mark.parametrize("layout", ["bhnd", "bnhd"])
@pytest.mark.parametrize("per_head", [False, True])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_plain_calls_are_marshalled_by_the_module(cpu_marshal, layout, per_head, dtype):
    """A plain call goes through with the addresses, sizes and variant word that binding.py gives; others are declined."""
    module, calls = cpu_marshal
    (B, H, N, d, k, m), (Q, K, V, E, F, W), dO = _small_call(layout, per_head, dtype)
    bnhd = layout == "bnhd"
    for variant, W1, m1 in ((PERFORMER, W, m), (RNN, None, 0)):
        word = binding._variant_word(variant, dtype, layout, per_head)
        ins = [t.data_ptr() for t in (Q, K, V, E, F)] + [W1.data_ptr() if W1 is not None else None]
        del calls[:]
        status, out = module.forward(Q, K, V, E, F, W1, variant, bnhd)
        assert status == 0 and out.shape == Q.shape and out.dtype == dtype
        assert calls == [(*ins, word, B, H, N, d, k, m1, out.data_ptr(), None)]
        del calls[:]
        status, *grads = module.backward(Q, K, V, E, F, W1, variant, bnhd, dO)
        assert status == 0 and [g.shape for g in grads] == [t.shape for t in (Q, K, V, E, F)]
        assert calls == [(*ins, dO.data_ptr(), word, B, H, N, d, k, m1, *[g.data_ptr() for g in grads], None)]
    del calls[:]
    other = torch.float32 if dtype is torch.bfloat16 else torch.bfloat16
    for bad in ((Q.transpose(1, 2), K, V, E, F, W), (Q, K.to(other), V, E, F, W), (Q, K[:1], V, E, F, W),
                (Q, K, V, E[..., :-1].contiguous(), F, W), (Q, K, V, E, F, W.t()), (Q, K, V, E, F, None), (None, K, V, E, F, W),
                (Q.as_subclass(_Subclass), K, V, E, F, W), [t.half() for t in (Q, K, V, E, F, W)]):
        assert module.forward(*bad, PERFORMER, bnhd) is None
        assert module.backward(*bad, PERFORMER, bnhd, dO) is None
    assert module.forward(Q, K, V, E, F, W, 7, bnhd) is None and module.forward(Q, K, V, E, F, W, True, bnhd) is None
    assert module.backward(Q, K, V, E, F, W, PERFORMER, bnhd, dO[:1]) is None
    assert not calls


@pytest.mark.parametrize("fault", ["built for another torch", "does not load"])
def test_library_works_without_the_marshalling_module(monkeypatch, fault):
    """No entry point depends on _marshal.so: the library loads with a warning, calls are checked and refused in Python."""
    build.build()
    if fault == "does not load":
        monkeypatch.setitem(sys.modules, "paper_2306_15799_b200._marshal", None)
        monkeypatch.delattr("paper_2306_15799_b200._marshal", raising=False)
    else:
        monkeypatch.setattr(build, "marshal_tag", lambda: b"marshalling for torch 0.0")
        assert not build.marshal_fits()
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_marshal", None)
    with pytest.warns(RuntimeWarning, match="_marshal.so"):
        binding.load()
    assert binding.version() == 100 and not binding._marshal.__name__.endswith("._marshal")
    _, args, dO = _small_call()
    with pytest.raises(ValueError):
        binding.flurka_forward(*args, PERFORMER)
    with pytest.raises(ValueError):
        binding.flurka_backward(*args, dO, PERFORMER)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("layout", ["bhnd", "bnhd"])
@pytest.mark.parametrize("per_head", [False, True])
def test_plain_calls_and_calls_with_outputs_agree(lib, dtype, layout, per_head):
    """A call without `out` and `stream` is marshalled in C++, the others in Python: same results, same refusals."""
    B, H, N, d, k, m = 2, 3, 72, 16, 8, 24
    gen = torch.Generator(device="cuda").manual_seed(5)
    r = lambda *s: torch.randn(*s, generator=gen, device="cuda").mul_(d ** -0.25).to(dtype)
    shape = (B, N, H, d) if layout == "bnhd" else (B, H, N, d)
    Q, K, V, dO = r(*shape), r(*shape), r(*shape), r(*shape)
    E, F = (r(H, k, N), r(H, k, N)) if per_head else (r(k, N), r(k, N))
    for variant, W in ((PERFORMER, r(m, d)), (RNN, None)):
        args = (Q, K, V, E, F, W, variant)
        assert binding._marshal.forward(*args, layout == "bnhd")[0] == 0
        out = binding.flurka_forward(*args, layout=layout)
        want = binding.flurka_forward(*args, layout=layout, out=torch.empty_like(Q))
        grads = binding.flurka_backward(Q, K, V, E, F, W, dO, variant, layout=layout)
        want_grads = binding.flurka_backward(Q, K, V, E, F, W, dO, variant, layout=layout,
                                             out=[torch.empty_like(t) for t in (Q, K, V, E, F)])
        torch.cuda.synchronize()
        # partial sums meet in any order, and bf16 results may round to either side of that
        tol = 1e-5 if dtype is torch.float32 else 4e-3
        for a, b in zip((out, *grads), (want, *want_grads)):
            assert a.shape == b.shape and a.dtype == b.dtype and a.is_contiguous()
            assert float((a.double() - b.double()).norm()) <= tol * float(b.double().norm())
        # a Parameter is a tensor too
        p = torch.nn.Parameter(Q.clone(), requires_grad=False)
        again = binding.flurka_forward(p, *args[1:], layout=layout)
        assert float((again.double() - want.double()).norm()) <= tol * float(want.double().norm())
    W = r(m, d)
    other = torch.float32 if dtype is torch.bfloat16 else torch.bfloat16
    for bad, kind in (((Q.cpu(), K, V, E, F, W), ValueError), ((Q.transpose(1, 2), K, V, E, F, W), ValueError),
                      ((Q, K.to(other), V, E, F, W), TypeError), ((Q, K[:1], V, E, F, W), ValueError),
                      ((Q, K, V, E[..., :-1].contiguous(), F, W), ValueError), ((Q, K, V, E, F, W.t()), ValueError),
                      ((Q, K, V, E, F, None), ValueError), ((Q.half(), K.half(), V.half(), E.half(), F.half(), W.half()), TypeError)):
        with pytest.raises(kind):
            binding.flurka_forward(*bad, PERFORMER, layout=layout)
        with pytest.raises(kind):
            binding.flurka_backward(*bad, dO, PERFORMER, layout=layout)
    with pytest.raises(binding.FlurkaError) as ei:
        binding.flurka_forward(Q, K, V, E, F, W, 7, layout=layout)
    assert ei.value.code == -2
    with pytest.raises(ValueError):
        binding.flurka_forward(Q, K, V, E, F, W, PERFORMER, layout="nbhd")
    with pytest.raises(RuntimeError):
        torch.func.vmap(lambda q: binding.flurka_forward(q, K, V, E, F, W, PERFORMER, layout=layout))(torch.stack([Q, Q]))
    for q, do in ((Q, dO), (dO, Q)):
        with pytest.raises(RuntimeError):
            torch.func.grad(lambda x: binding.flurka_backward(x, K, V, E, F, W, do, PERFORMER, layout=layout)[0].sum())(q)
