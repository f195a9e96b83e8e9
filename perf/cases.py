"""The work that is timed: what a program built on this library has it do, one public call sequence per case.

Shapes are those of the benchmark configurations (``paper_2407_12077_b200.synth.CONFIGS``: the D = 768 and D = 2048
models, long context, the serving mix) or generic ones beside them; values have the distributions of that module.
"""
from __future__ import annotations

import math

import torch

import paper_2407_12077_b200 as gf
from paper_2407_12077_b200 import synth

DEV = "cuda:0"
N = 64                                   # head size, the only one the library takes
STATE = N * N * 4                        # bytes of one (sequence, head) state


def listed():
    return [
        # one short prompt with everything in fp32: the smallest call, where latency is all there is
        dict(name="prefill-fp32", kind="prefill", form="classic", dtype="f32", B=1, T=256, H=4, state=False),
        # an interactive prompt through one layer of the D = 768 model, Finch-C2 form, no multiple of the chunk length
        dict(name="prompt", kind="prefill", form="c2", dtype="bf16", B=1, T=333, H=12, state=False),
        # batched prefill of the D = 768 model that continues from kept states
        dict(name="prefill-small-model", kind="prefill", form="classic", dtype="bf16", B=8, T=4096, H=12, state=True),
        # one layer's prefill of the D = 2048 (1.5B-class) model: the headline workload
        dict(name="prefill-1.5b", kind="prefill", form="classic", dtype="bf16", B=4, T=16384, H=32, state=False),
        # one long document, a single sequence
        dict(name="prefill-long", kind="prefill", form="classic", dtype="bf16", B=1, T=131072, H=32, state=False),
        # the Finch-C2 block from the recurrence to the norm before its output projection, ragged length
        dict(name="c2-output", kind="c2_output", B=5, T=2011, H=32, state=True),
        # batched serving: sequences of 128..4096 tokens packed into one call, each with its own start state
        dict(name="serving", kind="varlen", form="classic", S=64, lo=128, hi=4096, H=32),
        # one decode token for each of those sequences through the Finch-C2 layers of a 24-layer stack
        dict(name="decode", kind="decode", form="c2", S=64, H=32, layers=16),
        # a training step's pair at the paper's per-GPU batch (8 sequences of 2048 tokens), Finch-C2 form
        dict(name="train", kind="train", form="c2", B=8, T=2048, H=32, state=False),
        # the same pair over packed documents of uneven length, classic form
        dict(name="train-packed", kind="train_varlen", form="classic", S=24, lo=100, hi=3000, H=32),
        # the producer of the decay logits over the tokens of the headline prefill
        dict(name="decay-logit", kind="decay_logit", B=4, T=16384, H=32, Rd=32, Rw=64, prev=True),
        # the compressed key-cache entries of those tokens
        dict(name="key-compress", kind="key_compress", rows=65536, D=2048, Dc=128),
    ]


def _log(rng, lo, hi):
    """A whole number from lo..hi, spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["prefill", "prefill", "prefill-f32", "long", "c2_output", "varlen", "decode", "train", "train",
                       "train_varlen", "decay_logit", "key_compress"])
    form = rng.choice(["classic", "c2"])
    H = rng.choice([4, 12, 12, 20, 32, 32, 40])
    if kind == "prefill":
        T = _log(rng, 40, 16384)
        B = _log(rng, 1, max(1, min(64, 2_000_000 // (T * H))))
        return dict(kind="prefill", form=form, dtype="bf16", B=B, T=T, H=H, state=rng.random() < 0.5)
    if kind == "prefill-f32":
        return dict(kind="prefill", form="classic", dtype="f32", B=_log(rng, 1, 4), T=_log(rng, 40, 1024),
                    H=rng.choice([4, 12, 20]), state=rng.random() < 0.5)
    if kind == "long":                   # one or two long sequences
        B = rng.choice([1, 1, 2])
        return dict(kind="prefill", form=form, dtype="bf16", B=B, T=_log(rng, 16384, 131072 // B), H=rng.choice([12, 32]),
                    state=rng.random() < 0.5)
    if kind == "c2_output":
        T = _log(rng, 100, 8192)
        return dict(kind="c2_output", B=_log(rng, 1, max(1, min(32, 1_000_000 // (T * H)))), T=T, H=H, state=rng.random() < 0.5)
    if kind == "varlen":
        lo, hi = _log(rng, 32, 256), _log(rng, 512, 4096)
        return dict(kind="varlen", form=form, S=_log(rng, 2, 64), lo=lo, hi=hi, H=H)
    if kind == "decode":
        return dict(kind="decode", form=form, S=_log(rng, 1, 64), H=H if H < 40 else 32, layers=rng.randint(4, 16))
    if kind == "train":
        T = _log(rng, 200, 16384)
        return dict(kind="train", form=form, B=_log(rng, 1, max(1, min(16, 600_000 // (T * H)))), T=T, H=H,
                    state=rng.random() < 0.3)
    if kind == "train_varlen":
        return dict(kind="train_varlen", form=form, S=_log(rng, 4, 24), lo=_log(rng, 32, 200), hi=_log(rng, 400, 3000),
                    H=rng.choice([12, 32]))
    if kind == "decay_logit":
        T = _log(rng, 100, 16384)
        return dict(kind="decay_logit", B=_log(rng, 1, max(1, min(32, 65536 // T))), T=T, H=rng.choice([12, 20, 32]),
                    Rd=rng.choice([32, 32, 64]), Rw=64, prev=rng.random() < 0.5)
    D = rng.choice([768, 1280, 2048])
    return dict(kind="key_compress", rows=_log(rng, 200, 65536), D=D, Dc=D // 16)


def _seeded(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 1)


def _bf16(shape, gen, scale=1.0):
    return (torch.randn(shape, device=DEV, generator=gen) * scale).to(torch.bfloat16)


def _cu(case, seed):
    """Sequence boundaries of a packed batch: lengths spread evenly over lo..hi, in an order made from the seed."""
    S, lo, hi = case["S"], case["lo"], case["hi"]
    lens = lo + torch.div(torch.arange(S) * (hi - lo), max(1, S - 1), rounding_mode="floor")
    lens = lens[torch.randperm(S, generator=torch.Generator().manual_seed(int(seed)))]
    cu = torch.zeros(S + 1, dtype=torch.int32)
    cu[1:] = torch.cumsum(lens, 0).to(torch.int32)
    return cu


def _total(case):
    S, lo, hi = case["S"], case["lo"], case["hi"]
    return sum(lo + i * (hi - lo) // max(1, S - 1) for i in range(S))


def prepare(case, seed):
    kind, st = case["kind"], dict(case)
    gen = _seeded(seed)
    if kind in ("prefill", "c2_output", "train"):
        B, T, H = case["B"], case["T"], case["H"]
        st["in"] = synth.make_dense(B, T, H, N, case.get("dtype", "bf16"), seed=seed, device=DEV, state_std=0.1 if case["state"] else 0.0)
        if kind == "c2_output" or case["form"] == "c2":
            st["u2"] = _bf16((B, T, H, N), gen)
        if kind == "c2_output":
            st["gamma"] = 1 + 0.3 * torch.randn(H * N, device=DEV, generator=gen)
            st["beta"] = 0.2 * torch.randn(H * N, device=DEV, generator=gen)
        if kind == "train":
            st["dy"] = _bf16((B, T, H, N), gen)
            st["ws"] = torch.empty(gf.backward_workspace_bytes(B, T, H, N), dtype=torch.uint8, device=DEV)
    elif kind in ("varlen", "train_varlen"):
        cu, H = _cu(case, seed), case["H"]
        total = int(cu[-1])
        st["max"] = int((cu[1:] - cu[:-1]).max())
        st["in"] = synth.make_varlen(cu, H, N, "bf16", seed=seed, device=DEV, state_std=0.1)
        st["u2"] = _bf16((total, H, N), gen) if case["form"] == "c2" else None
        if kind == "train_varlen":
            st["dy"] = _bf16((total, H, N), gen)
            st["ws"] = torch.empty(gf.backward_varlen_workspace_bytes(case["S"], total, H, N), dtype=torch.uint8, device=DEV)
    elif kind == "decode":
        S, H = case["S"], case["H"]
        st["layers"] = [synth.make_step(S, H, N, "bf16", seed=1000 * seed + i, device=DEV) for i in range(case["layers"])]
        st["u2"] = [_bf16((S, H, N), gen) for _ in st["layers"]]
        st["y"] = [torch.empty_like(d.r) for d in st["layers"]]
        st["next"] = [torch.empty_like(d.state_in) for d in st["layers"]]    # states kept twice: this token's and the next one's
    elif kind == "decay_logit":
        D = case["H"] * N
        st["x"], st["xp"] = synth.make_block_input(case["B"], case["T"], D, seed=seed, device=DEV, with_prev=case["prev"])
        st["w"] = synth.make_decay_lora(D, case["Rd"], case["Rw"], seed=seed + 1, device=DEV)
    else:
        st["x"] = _bf16((case["rows"], case["D"]), gen)
        st["w"] = _bf16((case["D"], case["Dc"]), gen, case["D"] ** -0.5)
    return st


def run(st):
    kind, i = st["kind"], st.get("in")
    c2 = st.get("form") == "c2"
    if kind == "prefill":
        if c2:
            return gf.prefill_c2(i.r, i.k, i.v, i.x, st["u2"], i.state_in)
        return gf.prefill(i.r, i.k, i.v, i.x, i.u, i.state_in)
    if kind == "c2_output":
        y, s = gf.prefill_c2(i.r, i.k, i.v, i.x, st["u2"], i.state_in)
        return gf.layernorm_heads(y, st["gamma"], st["beta"], 1e-5), s
    if kind == "varlen":
        if c2:
            return gf.prefill_varlen_c2(i.r, i.k, i.v, i.x, st["u2"], i.cu_seqlens, st["max"], i.state_in)
        return gf.prefill_varlen(i.r, i.k, i.v, i.x, i.u, i.cu_seqlens, st["max"], i.state_in)
    if kind == "decode":
        for d, u2, y, nxt in zip(st["layers"], st["u2"], st["y"], st["next"]):
            if c2:
                gf.step_c2(d.r, d.k, d.v, d.x, u2, d.state_in, state_out=nxt, y=y)
            else:
                gf.step(d.r, d.k, d.v, d.x, d.u, d.state_in, state_out=nxt, y=y)
        return st["y"], st["next"]
    if kind == "train":
        y, s = gf.prefill_train(i.r, i.k, i.v, i.x, i.u, st["ws"], i.state_in, c2=c2, u2=st.get("u2"))
        if c2:
            return y, s, gf.backward_c2(i.r, i.k, i.v, i.x, st["dy"], i.state_in, workspace=st["ws"], saved=True)
        return y, s, gf.backward(i.r, i.k, i.v, i.x, i.u, st["dy"], i.state_in, workspace=st["ws"], saved=True)
    if kind == "train_varlen":
        y, s = gf.prefill_varlen_train(i.r, i.k, i.v, i.x, i.u, i.cu_seqlens, st["max"], st["ws"], i.state_in, c2=c2, u2=st["u2"])
        return y, s, gf.backward_varlen(i.r, i.k, i.v, i.x, i.u, st["dy"], i.cu_seqlens, st["max"], i.state_in,
                                        workspace=st["ws"], c2=c2, saved=True)
    if kind == "decay_logit":
        w = st["w"]
        return gf.decay_logit(st["x"], w["mu_x"], w["A_d"], w["B_d"], w["lambda_d"], w["A_w"], w["B_w"], w["lambda_w"], x_prev=st["xp"])
    return gf.key_compress(st["x"], st["w"])


def work(case):
    """Every input read once, every output written once.  Floating point: the recurrence itself (two multiply-adds per
    state element and token, six for its gradient), the products of the dense maps."""
    kind = case["kind"]
    if kind == "decay_logit":
        rows, D, R = case["B"] * case["T"], case["H"] * N, case["Rd"] + case["Rw"]
        return dict(bytes=4 * rows * D + 4 * D * R + 12 * D, flops=4 * rows * D * R)
    if kind == "key_compress":
        rows, D, Dc = case["rows"], case["D"], case["Dc"]
        return dict(bytes=2 * (rows * D + rows * Dc + D * Dc), flops=2 * rows * D * Dc)
    H = case["H"]
    if kind == "decode":
        units = case["layers"] * case["S"] * H
        return dict(bytes=units * (2 * STATE + 128 * (6 if case["form"] == "c2" else 5)), flops=4 * N * N * units)
    if kind in ("varlen", "train_varlen"):
        th, seqs, state = _total(case) * H, case["S"], True
    else:
        th, seqs, state = case["B"] * case["T"] * H, case["B"], case["state"]
    with_u2 = kind == "c2_output" or case["form"] == "c2"
    vec = 256 if case.get("dtype") == "f32" else 128
    nbytes = th * vec * (6 if with_u2 else 5) + seqs * H * STATE * (2 if state else 1)
    flops = 4 * N * N * th
    if kind in ("train", "train_varlen"):
        nbytes += th * vec * 9 + seqs * H * STATE * (2 if state else 1)
        flops *= 4
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    """About four times the relative error measured against the same path in float64 (largest over the outputs)."""
    kind = case["kind"]
    if kind == "prefill" and case["dtype"] == "f32":
        return {"rel": 1e-5}
    if kind == "decode":                 # fp32 state arithmetic; y is rounded to bf16 once
        return {"rel": 6e-3}
    if kind in ("decay_logit", "key_compress"):
        return {"rel": 7e-3}
    if kind in ("train", "train_varlen"):
        return {"rel": 1.5e-2}
    return {"rel": 1.3e-2}
