"""Dense calls with more (sequence, head) units than SMs whose units are cut between CTAs (balanced persistent launches).

The state at a cut is handed over in fp32 at a chunk boundary, so every result must equal, bit for bit, that of the same
sequences (of a single one: of its heads) run a part at a time without a cut (one CTA per unit); the smallest shapes are also
compared with the oracle."""
import pytest
import torch

import paper_2407_12077_b200 as gf
from oracle import wkv6_oracle as orc
from paper_2407_12077_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (B, T, H), on 148 SMs: 160 units of 5 ragged chunks; 222 of 11; 308 of 6 (one whole round, then the cut ones); 157 of 64
SHAPES = [(5, 300, 32), (3, 641, 74), (11, 321, 28), (1, 4096, 157)]


def parts(B, H):
    """Index pairs (sequences, heads) that cover a call in parts of few units: one sequence each, or halves of its heads.  Run
    with split=False (the gradient: with more than 74 units) a part takes one CTA per unit."""
    if B > 1:
        return [(slice(b, b + 1), slice(None)) for b in range(B)]
    return [(slice(None), slice(0, (H + 1) // 2)), (slice(None), slice((H + 1) // 2, H))]


@pytest.mark.parametrize("B,T,H", SHAPES)
@pytest.mark.parametrize("c2,in_place,x_hi", [(False, False, -1.0), (False, True, 2.5), (True, False, -1.0), (True, True, 2.5)])
def test_units_cut_between_ctas(B, T, H, c2, in_place, x_hi):
    # x_hi = 2.5: some chunks decay by more than 2^-96 and take the token-by-token path
    i = synth.make_dense(B, T, H, 64, "bf16", seed=B * T + H, device=DEV, state_std=0.1, x_hi=x_hi)
    u2 = torch.randn(i.r.shape, device=DEV, generator=torch.Generator(device=DEV).manual_seed(3)).bfloat16()

    def run(b, h, state, out=None, **kw):
        t = [x[b, :, h].contiguous() for x in (i.r, i.k, i.v, i.x, u2)]
        if c2:
            return gf.prefill_c2(*t, state, state_out=out, **kw)
        return gf.prefill(*t[:4], i.u[h].contiguous(), state, state_out=out, **kw)

    s0 = i.state_in.clone()
    y, s = run(slice(None), slice(None), s0, s0 if in_place else None)
    gf.last_device_status()
    for b, h in parts(B, H):
        yb, sb = run(b, h, i.state_in[b, h].contiguous(), split=False)
        assert torch.equal(yb, y[b, :, h]) and torch.equal(sb, s[b, h])
    gf.last_device_status()
    if T <= 321 and not c2:
        y_ref, s_ref = orc.prefill(*(t.cpu() for t in (i.r, i.k, i.v, i.x, i.u, i.state_in)))
        assert orc.rel_l2(y.float().cpu().numpy(), y_ref) <= 5e-3      # the contract's tolerance
        assert orc.rel_l2(s.cpu().numpy(), s_ref) <= 5e-3


@pytest.mark.parametrize("c2", [False, True])
def test_cut_call_repeats_and_replays(c2):
    # the announcement words lie in y: neither a reused y nor a replayed graph may see an old one
    i = synth.make_dense(5, 700, 32, 64, "bf16", seed=8, device=DEV, state_std=0.1)
    y, s = torch.empty_like(i.r), torch.empty_like(i.state_in)
    fn = (lambda st=None: gf.prefill_c2(i.r, i.k, i.v, i.x, i.r, i.state_in, state_out=s, y=y, stream=st)) if c2 else \
         (lambda st=None: gf.prefill(i.r, i.k, i.v, i.x, i.u, i.state_in, state_out=s, y=y, stream=st))
    fn()
    y0, s0 = y.clone(), s.clone()
    for _ in range(20):
        fn()
        assert torch.equal(y, y0) and torch.equal(s, s0)
    st, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=st):
            fn(st)
    for _ in range(5):
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, y0) and torch.equal(s, s0)
    gf.last_device_status()


@pytest.mark.parametrize("c2", [False, True])
@pytest.mark.parametrize("saved", [False, True])
def test_cut_gradient_replays_with_new_inputs(c2, saved):
    # a graph's launches carry the same arguments every time, and the workspace still holds the cuts' words and adjoints of the
    # replay before; token-by-token chunks in the units' later parts make the CTA that hands over the slower one
    B, T, H = 5, 641, 32

    def draw(seed):
        i = synth.make_dense(B, T, H, 64, "bf16", seed=seed, device=DEV, state_std=0.1)
        i.x[:, 2 * T // 3:, :, seed % 7::9] = 2.5
        return [i.r, i.k, i.v, i.x, i.u, i.state_in, torch.randn(i.r.shape, device=DEV, generator=torch.Generator(device=DEV).manual_seed(seed)).bfloat16()]

    def step(t, ws):
        r, k, v, x, u, s0, dy = t
        out = gf.prefill_train(r, k, v, x, u, ws, s0, c2=c2) if saved else ()
        if c2:
            return (*out, *gf.backward_c2(r, k, v, x, dy, s0, workspace=ws, saved=saved))
        return (*out, *gf.backward(r, k, v, x, u, dy, s0, workspace=ws, saved=saved))

    n = gf.backward_workspace_bytes(B, T, H, 64)
    held, ws, ws_eager = draw(20), torch.empty(n, dtype=torch.uint8, device=DEV), torch.empty(n, dtype=torch.uint8, device=DEV)
    step(held, ws)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = step(held, ws)
    for seed in (20, 21, 22, 23):
        for t, new in zip(held, draw(seed)):
            t.copy_(new)
        g.replay()
        torch.cuda.synchronize()
        gf.last_device_status()
        for a, b in zip(out, step(held, ws_eager)):
            assert torch.equal(a, b), seed
    gf.last_device_status()


@pytest.mark.parametrize("c2", [False, True])
@pytest.mark.parametrize("B,T,H", SHAPES[:3] + [(40, 90, 32)])
def test_training_forward_of_many_units(B, T, H, c2):
    # the checkpoints of cut (and, in the last shape, of streamed whole) units: the gradient from them equals the gradient
    # that makes its own
    i = synth.make_dense(B, T, H, 64, "bf16", seed=B + T + H, device=DEV, state_std=0.1)
    dy = torch.randn(i.r.shape, device=DEV, generator=torch.Generator(device=DEV).manual_seed(4)).bfloat16()
    ws = torch.empty(gf.backward_workspace_bytes(B, T, H, 64), dtype=torch.uint8, device=DEV)
    y, s = gf.prefill_train(i.r, i.k, i.v, i.x, i.u, ws, i.state_in, c2=c2)
    y1, s1 = (gf.prefill_c2(i.r, i.k, i.v, i.x, None, i.state_in) if c2 else gf.prefill(i.r, i.k, i.v, i.x, i.u, i.state_in))
    assert torch.equal(y, y1) and torch.equal(s, s1)
    back = (lambda **kw: gf.backward_c2(i.r, i.k, i.v, i.x, dy, i.state_in, **kw)) if c2 else \
           (lambda **kw: gf.backward(i.r, i.k, i.v, i.x, i.u, dy, i.state_in, **kw))
    for a, b in zip(back(workspace=ws, saved=True), back()):
        assert torch.equal(a, b)
    gf.last_device_status()


@pytest.mark.parametrize("c2", [False, True])
def test_packed_training_forward_as_a_stream(c2):
    # more units than SMs: the packed training forward walks units from a counter, empty sequences included
    lens = [0, 130, 64, 1, 700, 63, 0, 65, 200, 128]
    cu = torch.tensor([0] + torch.tensor(lens).cumsum(0).tolist(), dtype=torch.int32)
    i = synth.make_varlen(cu, 20, 64, "bf16", seed=11, device=DEV, state_std=0.1)
    total, S = int(cu[-1]), len(lens)
    u2 = i.v if c2 else None
    dy = torch.randn(i.r.shape, device=DEV, generator=torch.Generator(device=DEV).manual_seed(5)).bfloat16()
    ws = torch.empty(gf.backward_varlen_workspace_bytes(S, total, 20, 64), dtype=torch.uint8, device=DEV)
    y, s = gf.prefill_varlen_train(i.r, i.k, i.v, i.x, i.u, i.cu_seqlens, 700, ws, i.state_in, c2=c2, u2=u2)
    y1, s1 = (gf.prefill_varlen_c2(i.r, i.k, i.v, i.x, u2, i.cu_seqlens, 700, i.state_in) if c2 else
              gf.prefill_varlen(i.r, i.k, i.v, i.x, i.u, i.cu_seqlens, 700, i.state_in))
    assert torch.equal(y, y1) and torch.equal(s, s1)
    kw = dict(c2=c2)
    for a, b in zip(gf.backward_varlen(i.r, i.k, i.v, i.x, i.u, dy, i.cu_seqlens, 700, i.state_in, workspace=ws, saved=True, **kw),
                    gf.backward_varlen(i.r, i.k, i.v, i.x, i.u, dy, i.cu_seqlens, 700, i.state_in, **kw)):
        assert a is None and b is None or torch.equal(a, b)
    gf.last_device_status()


@pytest.mark.parametrize("B,T,H", SHAPES + [(6, 200, 32)])
@pytest.mark.parametrize("c2", [False, True])
@pytest.mark.parametrize("x_hi,with_dstate", [(-1.0, True), (2.5, False)])
def test_gradient_units_cut_between_ctas(B, T, H, c2, x_hi, with_dstate):
    # each part on its own (few units and short, or more than half the SMs: one CTA per unit) gives the same bits; the bonus
    # gradient, summed over the batch, to fp32 rounding of its B * T terms
    i = synth.make_dense(B, T, H, 64, "bf16", seed=B + 3 * T + H, device=DEV, state_std=0.1, x_hi=x_hi)
    g = torch.Generator(device=DEV).manual_seed(6)
    dy = torch.randn(i.r.shape, device=DEV, generator=g).bfloat16()
    ds = torch.randn(i.state_in.shape, device=DEV, generator=g) if with_dstate else None

    def grad(b, h):
        t = [x[b, :, h].contiguous() for x in (i.r, i.k, i.v, i.x)]
        kw = dict(state_in=i.state_in[b, h].contiguous(), dstate_out=None if ds is None else ds[b, h].contiguous(), want_dstate=with_dstate)
        if c2:
            return gf.backward_c2(*t, dy[b, :, h].contiguous(), **kw)
        return gf.backward(*t, i.u[h].contiguous(), dy[b, :, h].contiguous(), **kw)

    full = grad(slice(None), slice(None))
    du = torch.zeros_like(i.u, dtype=torch.float64)
    for b, h in parts(B, H):
        one = grad(b, h)
        for n in range(4):
            assert torch.equal(one[n], full[n][b, :, h]), (b, h, n)
        if with_dstate:
            assert torch.equal(one[-1], full[-1][b, h])
        if not c2:
            du[h] += one[4].double()
    if not c2:
        assert float((full[4].double() - du).norm() / du.norm()) < 1e-5
    gf.last_device_status()


@pytest.mark.parametrize("T,c2", [(1025, True), (1025, False), (4100, False)])
def test_gradient_where_an_eighth_of_the_last_round_is_idle(T, c2):
    # 240 units on 148 SMs, 0.19 of the last round idle: units of 17 and 65 chunks are cut there; a sequence alone has more units than
    # half the SMs, one CTA each
    test_gradient_units_cut_between_ctas(3, T, 80, c2, -1.0, True)
