"""The binding's C++ part (csrc/binding.cpp) against the Python code it takes the place of: the same outputs for the plain form of
a call, and for every other form what Python makes of it."""
import os

import pytest
import torch

import paper_2407_12077_b200 as gf
from paper_2407_12077_b200 import _build, synth

DEV = "cuda:0"


@pytest.fixture
def both(monkeypatch):
    """Runs a call with the C++ part and without it: [result or (exception type, text)] of each."""
    gf.load_library()
    native = gf._native

    def run(fn):
        out = []
        for n in (native, None):
            monkeypatch.setattr(gf, "_native", n)
            try:
                out.append(fn())
            except Exception as e:
                out.append((type(e), str(e)))
        monkeypatch.setattr(gf, "_native", native)
        return out

    return run


def test_leaves_what_is_not_on_the_current_device_to_python():
    gf.load_library()
    if gf._native is None:
        assert not os.path.exists(_build.BINDING_PATH)       # (no compiler here: the Python code does without)
        pytest.skip("not built")
    t, u = torch.zeros(1, 4, 1, 64), torch.zeros(1, 64)
    for args in ((t, t, t, t, u, None, False), (None,) * 7, (1, 2, 3, 4, 5, 6, True), (t,)):
        assert gf._native.prefill(*args) is None
    assert gf._native.step(*[torch.zeros(1, 1, 64)] * 4, u, None, u, t, False) is None
    assert gf._native.layernorm(t, None, None, 1e-5) is None and gf._native.key_compress(t, t) is None
    assert gf._native.prefill_varlen(t, t, t, t, u, t, 4, None, False) is None
    with pytest.raises(ValueError, match="CUDA tensor"):
        gf.prefill(t, t, t, t, u)


def flat(o):
    return [t for x in (o if isinstance(o, (tuple, list)) else [o]) for t in (x if isinstance(x, (tuple, list)) else [x])]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_same_results(both, dtype):
    assert gf._native is not None or gf.load_library() and gf._native is not None
    i = synth.make_dense(2, 70, 3, 64, dtype, seed=1, device=DEV, state_std=0.1)
    p = synth.make_varlen(torch.tensor([0, 5, 5, 90], dtype=torch.int32), 3, 64, dtype, seed=2, device=DEV, state_std=0.1)
    s = synth.make_step(3, 2, 64, dtype, seed=3, device=DEV)
    g, b = torch.randn(192, device=DEV), torch.randn(192, device=DEV)
    calls = [lambda: gf.prefill(i.r, i.k, i.v, i.x, i.u), lambda: gf.prefill(i.r, i.k, i.v, i.x, torch.nn.Parameter(i.u), i.state_in),
             lambda: gf.prefill(i.r.clone().requires_grad_(), i.k, i.v, i.x, i.u, i.state_in),
             lambda: gf.prefill_varlen(p.r, p.k, p.v, p.x, p.u, p.cu_seqlens, 85, p.state_in), lambda: gf.step(s.r, s.k, s.v, s.x, s.u, s.state_in.clone()),
             lambda: gf.step(s.r, s.k, s.v, s.x, s.u, None), lambda: gf.layernorm_heads(i.r, g, b, 1e-5), lambda: gf.layernorm_heads(i.r, g.view(3, 64))]
    if dtype == "bf16":
        w = torch.randn(192, 64, device=DEV).bfloat16()
        calls += [lambda: gf.prefill_c2(i.r, i.k, i.v, i.x), lambda: gf.prefill_c2(i.r, i.k, i.v, i.x, i.k, i.state_in),
                  lambda: gf.prefill_varlen_c2(p.r, p.k, p.v, p.x, p.k, p.cu_seqlens, 85, p.state_in), lambda: gf.step_c2(s.r, s.k, s.v, s.x, None, s.state_in.clone()),
                  lambda: gf.key_compress(i.r.view(2, 70, 192), w)]
    for n, call in enumerate(calls):
        a, b_ = both(call)
        for x, y in zip(flat(a), flat(b_), strict=True):
            assert torch.equal(x, y) and x.stride() == y.stride() and x.dtype == y.dtype and not x.requires_grad and not y.requires_grad, n
    gf.last_device_status()


@pytest.mark.gpu
def test_other_forms_are_what_python_makes_of_them(both):
    from torch._subclasses.fake_tensor import FakeTensorMode
    i = synth.make_dense(2, 70, 3, 64, "bf16", seed=1, device=DEV, state_std=0.1)
    s = synth.make_step(3, 2, 64, "bf16", seed=3, device=DEV)
    t = (i.k, i.v, i.x, i.u)
    wide = torch.zeros(2, 70, 3, 128, device=DEV, dtype=torch.bfloat16)
    refused = [lambda: gf.prefill(i.r, wide[..., :64], i.v, i.x, i.u), lambda: gf.prefill(i.r, i.k.float(), i.v, i.x, i.u), lambda: gf.prefill(i.r, i.k[:1], i.v, i.x, i.u),
               lambda: gf.prefill(i.r, i.k.cpu(), i.v, i.x, i.u), lambda: gf.prefill(i.r, *t[:3], i.u.bfloat16()), lambda: gf.prefill(i.r, *t[:3], None),
               lambda: gf.prefill(i.r, *t, i.state_in[:1]), lambda: gf.prefill(i.r[0], *t), lambda: gf.prefill(i.r.half(), *t), lambda: gf.prefill(wide, wide, wide, wide, torch.zeros(3, 128, device=DEV)),
               lambda: gf.step(s.r, s.k, s.v, s.x, s.u, s.state_in[:1]), lambda: gf.step(s.r, s.k, s.v, s.x, s.u, s.state_in, y=s.r), lambda: gf.step(s.r[0], s.k, s.v, s.x, s.u, None),
               lambda: gf.layernorm_heads(i.r, torch.zeros(191, device=DEV)), lambda: gf.key_compress(i.r, i.r[0, 0]),
               lambda: torch.vmap(lambda r: gf.prefill(r, *t))(i.r[None])]
    with FakeTensorMode(allow_non_fake_inputs=True) as mode:
        fake = mode.from_tensor(i.r)
    refused.append(lambda: gf.prefill(fake, *t))
    for n, call in enumerate(refused):
        a, b = both(call)
        assert isinstance(a, tuple) and isinstance(a[0], type) and a == b, (n, a, b)
    # a dispatch mode sees the allocations of both
    from torch.utils._python_dispatch import TorchDispatchMode

    class Names(TorchDispatchMode):
        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            self.seen.append(str(func))
            return func(*args, **(kwargs or {}))

    def seen():
        with Names() as m:
            m.seen = []
            gf.prefill(i.r, *t)
        return m.seen

    a, b = both(seen)
    assert a == b and a
    # a captured call takes its outputs from the graph's pool and its stream from the capture
    gf.prefill(i.r, *t)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        y, _ = gf.prefill(i.r, *t)
    y.zero_()
    graph.replay()
    assert torch.equal(y, gf.prefill(i.r, *t)[0])
    gf.last_device_status()
