"""Split calls (few (sequence, head) units) whose summary launch may start late in its segments: decays on both sides of
the threshold, and non-finite inputs before the point where it starts."""
import pytest
import torch

import paper_2407_12077_b200 as gf
from oracle import wkv6_oracle as orc
from paper_2407_12077_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
NAN, INF = float("nan"), float("inf")


@pytest.mark.parametrize("T", [24576, 25000, 66560, 66700])
@pytest.mark.parametrize("x_lo,x_hi", [(-6.0, -1.0), (-4.5, -4.0), (-5.4, -5.1), (-7.0, -6.5), (-1.0, -0.5), (-3.6, -3.2), (-3.4, -3.0)])
def test_late_start_against_oracle(T, x_lo, x_hi):
    # about 42 / 210 / 580 / 2600 / 7 / 90 / 74 chunks until every channel has decayed by 2^-280: from the first look of 15
    # chunks to the sixth, and beyond; segments of 48 and 49 chunks, which do not start late, of 130 and 131.  One
    # slow channel in head 1.  Tolerance: the contract's.
    inp = synth.make_dense(1, T, 3, 64, "bf16", seed=T, state_std=1.0, x_lo=x_lo, x_hi=x_hi)
    inp.x[:, :, 1, 17] = -11.0
    d = inp.to(DEV)
    assert gf.workspace_bytes(1, T, 3, 64) > 0
    y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    gf.last_device_status()
    y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    for h in range(3):
        assert orc.rel_l2(y[:, :, h].float().cpu().numpy(), y_ref[:, :, h]) <= 5e-3
        assert orc.rel_l2(s[:, h].cpu().numpy(), s_ref[:, h]) <= 5e-3


@pytest.mark.parametrize("log2_kv,chunks", [(0, 20), (0, 23), (100, 30), (100, 36), (100, 41)])
def test_what_lies_before_an_empty_tail_is_kept(log2_kv, chunks):
    # the keys and values of the segments' last chunks are zero, every channel decays by about 2^-5.6 in each of them, and the
    # last segment, without keys and without decay, hands the state on: what the tails leave of k v 2^log2_kv, down to
    # 2^-130, is the whole of it.  Against the unsplit call, whose products are the same and whose sums differ in what a segment
    # starts from: fp32 rounding of the sums of a channel's row, twice 2^-24 in each of the segment's chunks, and a subnormal.
    H, seg = 4, 128
    T = 8 * seg * 64
    assert gf.split_plan(1, T, H, torch.cuda.get_device_properties(0).multi_processor_count)[:2] == (8, seg)
    i = synth.make_dense(1, T, H, 64, "bf16", seed=31, device=DEV)
    i.x.copy_((-2.735 + 0.02 * i.x.float()).bfloat16())                      # (x around -3.5, so about -2.8)
    for t in (i.k, i.v):
        t.mul_(2.0 ** (log2_kv / 2))
        t.view(8, seg * 64, H, 64)[:, (seg - chunks) * 64:] = 0
    for t, value in ((i.k, 0), (i.v, 0), (i.x, -30)):
        t[:, 7 * seg * 64:] = value
    y, s = gf.prefill(i.r, i.k, i.v, i.x, i.u, None)
    y1, s1 = gf.prefill(i.r, i.k, i.v, i.x, i.u, None, split=False)
    gf.last_device_status()
    assert int((s1 != 0).sum()) > 0.99 * s1.numel()
    assert bool(((s - s1).abs() <= 2 * seg * 2.0 ** -24 * s1.abs().amax(-1, keepdim=True) + 2.0 ** -149).all())


@pytest.mark.parametrize("c2", [False, True])
@pytest.mark.parametrize("train", [False, True])
@pytest.mark.parametrize("T", [24576, 69632])
def test_non_finite_values_are_not_forgotten(T, c2, train):
    # one call per place: the tokens after it and the final state are non-finite where the unsplit call's are, the other
    # head is untouched (segments of 48 chunks, which do not start late, and of 136)
    H = 2
    clean = synth.make_dense(1, T, H, 64, "bf16", seed=5, device=DEV, state_std=0.1)
    ws = torch.empty(gf.backward_workspace_bytes(1, T, H, 64), dtype=torch.uint8, device=DEV)

    def run(i, split):
        if train and split:
            return gf.prefill_train(i.r, i.k, i.v, i.x, i.u, ws, i.state_in, c2=c2)
        if c2:
            return gf.prefill_c2(i.r, i.k, i.v, i.x, None, i.state_in, split=split)
        return gf.prefill(i.r, i.k, i.v, i.x, i.u, i.state_in, split=split)

    y0, s0 = run(clean, True)
    for name, t, value in [("k", 70, NAN), ("v", 4500, NAN), ("x", 9000, NAN), ("v", 10, INF), ("k", 6300, INF), ("v", T - 700, NAN)]:
        i = synth.make_dense(1, T, H, 64, "bf16", seed=5, device=DEV, state_std=0.1)
        getattr(i, name)[0, t, 1, 9] = value
        y, s = run(i, True)
        y1, s1 = run(i, False)
        gf.last_device_status()
        assert torch.equal(y[:, :, 0], y0[:, :, 0]) and torch.equal(s[:, 0], s0[:, 0]), name
        bad, bad1 = ~torch.isfinite(y[0, :, 1]), ~torch.isfinite(y1[0, :, 1])
        assert torch.equal(bad.any(1), bad1.any(1)), (name, t)               # the same tokens
        assert bool((bad | ~bad1).all()), (name, t)                          # and at least the same elements
        sb, sb1 = ~torch.isfinite(s[0, 1]), ~torch.isfinite(s1[0, 1])
        assert bool((sb | ~sb1).all()), (name, t)
        if train:                            # the states the gradient takes from the forward pass: as those it makes itself
            back = (lambda **kw: gf.backward_c2(i.r, i.k, i.v, i.x, i.r, i.state_in, **kw)) if c2 else \
                   (lambda **kw: gf.backward(i.r, i.k, i.v, i.x, i.u, i.r, i.state_in, **kw))
            for a, b in zip(back(workspace=ws, saved=True), back()):
                assert bool((~torch.isfinite(a) | torch.isfinite(b)).all()), (name, t)        # non-finite wherever the other is
                if a.dim() == 4 and a.shape[1] == T:
                    assert bool(torch.isfinite(a[:, :, 0]).all()), (name, t)
            gf.last_device_status()
    y, s = run(clean, True)                                                  # nothing stays behind
    assert torch.equal(y, y0) and torch.equal(s, s0)
