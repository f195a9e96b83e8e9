"""GPU parity: the CUDA library (called through its C ABI) against the fp64 CPU oracle on
the same seeded inputs.  Tolerances are the contract's: relative L2 <= 1e-4 for fp32
inputs, <= 5e-3 for bf16 inputs with fp32 state, on the outputs and on the final state.
"""
import numpy as np
import pytest
import torch

import paper_2407_12077_b200 as gf
from oracle import wkv6_oracle as orc
from paper_2407_12077_b200 import synth

pytestmark = pytest.mark.gpu

TOL = {torch.float32: 1e-4, torch.bfloat16: 5e-3}
DEV = "cuda:0"
KERNELS = {"exact": gf.KERNEL_EXACT, "chunked": gf.KERNEL_CHUNKED, "auto": gf.KERNEL_AUTO}


@pytest.fixture(autouse=True)
def _reset_kernel():
    yield
    gf.set_kernel(gf.KERNEL_AUTO)
    gf.last_device_status()


def check(y_gpu, s_gpu, y_ref, s_ref, tol, what=""):
    ey = orc.rel_l2(y_gpu.float().cpu().numpy(), y_ref)
    assert np.isfinite(ey) and ey <= tol, f"{what} y rel-L2 {ey:.3e} > {tol}"
    if s_gpu is not None:
        es = orc.rel_l2(s_gpu.cpu().numpy(), s_ref)
        assert np.isfinite(es) and es <= tol, f"{what} state rel-L2 {es:.3e} > {tol}"
        return ey, es
    return ey, None


def run_dense(inp, kernel="auto"):
    gf.set_kernel(KERNELS[kernel])
    d = inp.to(DEV)
    y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    gf.last_device_status()
    return y, s


def dense_case(B, T, H, dtype, seed, state_std, kernel, **kw):
    inp = synth.make_dense(B, T, H, 64, dtype, seed=seed, state_std=state_std, **kw)
    y, s = run_dense(inp, kernel)
    y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    return check(y, s, y_ref, s_ref, TOL[inp.r.dtype], f"B{B} T{T} H{H} {dtype} {kernel}")


def test_cfg0_fp32_full():
    c = synth.CONFIGS["cfg0"]
    dense_case(c["B"], c["T"], c["H"], "f32", seed=0, state_std=0.0, kernel="auto")


@pytest.mark.parametrize("T", [1, 2, 15, 16, 17, 63, 64, 65, 127, 128, 129, 200, 321])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_exact_kernel_ragged_lengths(T, dtype):
    dense_case(2, T, 3, dtype, seed=100 + T, state_std=0.1, kernel="exact")


@pytest.mark.parametrize("B,H", [(1, 18), (1, 19), (2, 37), (3, 25)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_exact_kernel_column_slabs(B, H, dtype):
    # units on both sides of the slab rule (eight, four or one CTA per unit on a GPU of 148 SMs); two tiles plus a token.
    # Tolerance: the contract's.
    dense_case(B, 33, H, dtype, seed=140 + B * H, state_std=0.1, kernel="exact")


@pytest.mark.parametrize("T", [1, 2, 15, 16, 17, 63, 64, 65, 127, 128, 129, 200, 321, 1000])
@pytest.mark.parametrize("state_std", [0.0, 0.1])
def test_chunked_kernel_ragged_lengths(T, state_std):
    dense_case(2, T, 3, "bf16", seed=200 + T, state_std=state_std, kernel="chunked")


@pytest.mark.parametrize("kernel", ["exact", "chunked"])
def test_cfg1_small_model_shape_full(kernel):
    c = synth.CONFIGS["cfg1"]
    dense_case(c["B"], c["T"], c["H"], "bf16", seed=1000, state_std=c["state_std"], kernel=kernel)


TOK_TOL = 4e-2      # supplementary per-token bound for bf16 inputs, see check_units


def check_units(y_gpu, s_gpu, y_ref, s_ref, what, tol=5e-3, tok_tol=TOK_TOL):
    """Dense [B,T,H,N] outputs and [B,H,N,N] states against the oracle: the contract's relative L2 over the whole
    tensors AND for every (b,h) unit on its own, plus a per-token bound on y that a norm over 16384 tokens cannot
    give: max over tokens of ||y_gpu[t] - y_ref[t]||_2 over the unit's r.m.s. row norm (a corrupted row must not
    hide behind a long sequence).  Returns the worst figures."""
    yg = y_gpu.float().cpu().numpy() if hasattr(y_gpu, "cpu") else y_gpu
    sg = s_gpu.cpu().numpy() if hasattr(s_gpu, "cpu") else s_gpu
    assert np.isfinite(yg).all() and np.isfinite(sg).all(), what
    T = yg.shape[1]
    d = yg - y_ref
    row = (d * d).sum(axis=3)                                  # [B,T,H] squared row errors
    num, den = row.sum(axis=1), (y_ref * y_ref).sum(axis=(1, 3))   # [B,H]
    whole = float(np.sqrt(num.sum() / den.sum()))
    unit = np.sqrt(num / den)
    tok = np.sqrt(row.max(axis=1) / (den / T))
    ds = sg - s_ref
    snum, sden = (ds * ds).sum(axis=(2, 3)), (s_ref * s_ref).sum(axis=(2, 3))
    swhole, sunit = float(np.sqrt(snum.sum() / sden.sum())), np.sqrt(snum / sden)
    assert whole <= tol and swhole <= tol, f"{what}: y {whole:.3e} state {swhole:.3e} > {tol}"
    assert unit.max() <= tol, f"{what}: unit {np.unravel_index(unit.argmax(), unit.shape)} y rel-L2 {unit.max():.3e} > {tol}"
    assert sunit.max() <= tol, f"{what}: unit {np.unravel_index(sunit.argmax(), sunit.shape)} state rel-L2 {sunit.max():.3e} > {tol}"
    assert tok.max() <= tok_tol, f"{what}: unit {np.unravel_index(tok.argmax(), tok.shape)} worst token {tok.max():.3e} > {tok_tol}"
    return whole, swhole, float(unit.max()), float(sunit.max()), float(tok.max())


@pytest.mark.parametrize("seed", [2000, 2007, 2015])
def test_cfg2_full_size_every_unit(seed):
    """1.5B-class shape at full size in the launch configuration the benchmark times (three of its sixteen
    independently seeded calls): all 128 (b,h) units and every token against the oracle."""
    c = synth.CONFIGS["cfg2"]
    inp = synth.make_dense(c["B"], c["T"], c["H"], 64, "bf16", seed=seed, device=DEV)
    gf.set_kernel(gf.KERNEL_AUTO)
    before = gf.launch_count()
    y, s = gf.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, None)
    gf.last_device_status()
    assert gf.launch_count() - before == 1
    cpu = inp.to("cpu")
    y_ref, s_ref = orc.prefill(cpu.r, cpu.k, cpu.v, cpu.x, cpu.u, None)
    print("cfg2", seed, check_units(y, s, y_ref, s_ref, f"cfg2 seed {seed}"))


def test_cfg3_long_context_every_head_in_segments_and_as_one_call():
    """T = 131072 as 8 segments of 16384 with state_out fed to the next state_in (in place), and as one call that
    the library splits itself, must both equal the unsegmented oracle: all 32 heads, every token."""
    c = synth.CONFIGS["cfg3"]
    T, H, nseg = c["T"], c["H"], c["segments"]
    inp = synth.make_dense(1, T, H, 64, "bf16", seed=3000, device=DEV)
    cpu = inp.to("cpu")
    y_ref, s_ref = orc.prefill(cpu.r, cpu.k, cpu.v, cpu.x, cpu.u, None)
    seg = T // nseg
    state = torch.zeros((1, H, 64, 64), device=DEV)
    y = torch.empty_like(inp.r)
    for i in range(nseg):
        sl = slice(i * seg, (i + 1) * seg)
        gf.prefill(inp.r[:, sl], inp.k[:, sl], inp.v[:, sl], inp.x[:, sl], inp.u, state, state_out=state, y=y[:, sl])
    gf.last_device_status()
    print("cfg3 segments", check_units(y, state, y_ref, s_ref, "cfg3 as 8 segment calls"))
    before = gf.launch_count()
    y1, s1 = gf.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, None)
    gf.last_device_status()
    assert gf.launch_count() - before == 2                       # summary launch + main launch
    print("cfg3 one call", check_units(y1, s1, y_ref, s_ref, "cfg3 as one call"))


@pytest.mark.parametrize("B,T,H,state_std,x_hi", [
    (1, 64 * 16 + 37, 2, 0.1, -1.0),     # 2 segments, ragged tail in the last
    (1, 5000, 4, 0.0, -1.0),             # 8 segments of 10 chunks, the last shorter
    (2, 3000, 3, 0.1, -1.0),             # 6 units
    (1, 1100, 2, 0.1, 3.0),              # strong decay: token-by-token chunks inside both passes
])
def test_sequence_split_matches_oracle_and_unsplit_call(B, T, H, state_std, x_hi):
    """Few (b,h) units: the call cuts every sequence into segments (summary launch + main launch over a
    scratch workspace).  Same result as the oracle, and as the single-launch path to rounding."""
    assert gf.workspace_bytes(B, T, H, 64) > 0, "this shape is expected to split"
    inp = synth.make_dense(B, T, H, 64, "bf16", seed=1234 + T, state_std=state_std, x_lo=-6.0 if x_hi < 0 else -1.0, x_hi=x_hi)
    d = inp.to(DEV)
    gf.set_kernel(gf.KERNEL_CHUNKED)
    before = gf.launch_count()
    y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    assert gf.launch_count() - before == 2
    y1, s1 = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in, split=False)
    assert gf.launch_count() - before == 3
    y2, s2 = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    gf.last_device_status()
    assert torch.equal(y, y2) and torch.equal(s, s2)                 # deterministic, workspace reuse is clean
    y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    check(y, s, y_ref, s_ref, 5e-3, "split")
    check(y1, s1, y_ref, s_ref, 5e-3, "unsplit")
    assert orc.rel_l2(y.float().cpu().numpy(), y1.float().cpu().numpy()) < 2e-3
    assert orc.rel_l2(s.cpu().numpy(), s1.cpu().numpy()) < 1e-3


@pytest.mark.parametrize("B,T,H", [(1, 5000, 4), (1, 16384, 32), (2, 3000, 3)])
def test_sequence_split_with_the_state_updated_in_place(B, T, H):
    """state_out == state_in under the sequence split: the first launch keeps a copy of the start states in the
    scratch and the second launch reads only the copy, so no CTA can find the final state where it expects the
    start state.  Slow decays (w about 0.9999), so that the start state reaches the last token and the final state."""
    assert gf.workspace_bytes(B, T, H, 64) > 0
    inp = synth.make_dense(B, T, H, 64, "bf16", seed=1300 + T, state_std=2.0, x_lo=-12.0, x_hi=-8.0)
    d = inp.to(DEV)
    gf.set_kernel(gf.KERNEL_CHUNKED)
    y0, s0 = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    st = d.state_in.clone()
    before = gf.launch_count()
    y1, s1 = gf.prefill(d.r, d.k, d.v, d.x, d.u, st, state_out=st)
    gf.last_device_status()
    assert gf.launch_count() - before == 2 and s1.data_ptr() == st.data_ptr()
    assert torch.equal(y0, y1) and torch.equal(s0, st)
    y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    check_units(y1, st, y_ref, s_ref, f"in-place split B{B} T{T} H{H}")
    # the start state matters in this test: a zero start misses the final state by twice the tolerance or more
    y_z, s_z = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, None)
    assert orc.rel_l2(s_z, s_ref) > 1e-2


def test_packed_sequence_split_with_the_state_updated_in_place():
    """The same for a packed call cut by max_seqlen, where the shorter sequence's last segments are empty (their CTAs
    only fold the summaries and write the final state at once)."""
    lens, H = [3000, 700, 0], 4
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32)
    assert gf.workspace_bytes(len(lens), max(lens), H, 64) > 0
    inp = synth.make_varlen(cu, H, 64, "bf16", seed=1400, state_std=0.5, x_lo=-12.0, x_hi=-8.0)
    d = inp.to(DEV)
    gf.set_kernel(gf.KERNEL_CHUNKED)
    y0, s0 = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, max(lens), d.state_in)
    st = d.state_in.clone()
    before = gf.launch_count()
    y1, _ = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, max(lens), st, state_out=st)
    gf.last_device_status()
    assert gf.launch_count() - before == 2
    assert torch.equal(y0, y1) and torch.equal(s0, st)
    y_ref, s_ref = orc.prefill_varlen(inp.r, inp.k, inp.v, inp.x, inp.u, cu, inp.state_in)
    check(y1, st, y_ref, s_ref, 5e-3, "in-place packed split")
    for i, n in enumerate(lens):
        a, b = int(cu[i]), int(cu[i + 1])
        if n:
            check(y1[a:b], st[i], y_ref[a:b], s_ref[i], 5e-3, f"in-place packed split seq {i}")
        else:
            assert torch.equal(st[i].cpu(), inp.state_in[i])


def test_random_shapes_and_decay_patterns_against_oracle():
    """Seeded sweep over lengths (all residues of the ring and buffer depths), unit counts, initial states and
    decay patterns, including sequences where only some chunks decay too fast for the tensor-core path."""
    import random
    rng = random.Random(20240712)
    gf.set_kernel(gf.KERNEL_CHUNKED)
    for it in range(36):
        B, H = rng.choice([1, 1, 2, 3]), rng.choice([1, 2, 3, 5])
        T = rng.choice([rng.randint(1, 700), 64 * rng.randint(1, 14), 64 * rng.randint(1, 12) + 1, rng.randint(700, 1500)])
        mode = rng.choice(["plain", "plain", "fast", "mixed", "patchy"])
        inp = synth.make_dense(B, T, H, 64, "bf16", seed=5000 + it, state_std=rng.choice([0.0, 0.1]))
        g = torch.Generator().manual_seed(6000 + it)
        if mode == "fast":
            inp.x = (torch.rand(inp.x.shape, generator=g) * 4 - 1).bfloat16()
        elif mode == "mixed":
            inp.x = (torch.rand(inp.x.shape, generator=g) * 16 - 8).bfloat16()
        elif mode == "patchy":
            xf = inp.x.float()
            for c in range(0, T, 64):
                if rng.random() < 0.3:
                    xf[:, c:c + 64] = torch.rand(xf[:, c:c + 64].shape, generator=g) * 3 + 0.5
            inp.x = xf.bfloat16()
        d = inp.to(DEV)
        y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in, split=rng.choice([True, False]))
        gf.last_device_status()
        y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
        assert torch.isfinite(y.float()).all() and torch.isfinite(s).all()
        check(y, s, y_ref, s_ref, 5e-3, f"case {it}: B{B} T{T} H{H} {mode}")


def test_quarter_million_tokens_one_head():
    """One (b,h) unit of 262144 tokens: 4096 chunks cut into 8 segments (every barrier phase and ring slot
    wraps hundreds of times); the fp32 state must stay on the oracle's over the whole length."""
    T = 262144
    inp = synth.make_dense(1, T, 1, 64, "bf16", seed=7000, device=DEV)
    assert gf.workspace_bytes(1, T, 1, 64) == (7 * (64 + 4096) + 4096) * 4      # 7 summaries + the start-state copy
    gf.set_kernel(gf.KERNEL_CHUNKED)
    y, s = gf.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, None)
    gf.last_device_status()
    cpu = inp.to("cpu")
    y_ref, s_ref = orc.prefill(cpu.r, cpu.k, cpu.v, cpu.x, cpu.u, None)
    check(y, s, y_ref, s_ref, 5e-3, "T=262144")
    # and the tail of the sequence on its own, where an error in a carried state would show
    check(y[:, -4096:], None, y_ref[:, -4096:], None, 5e-3, "last 4096 tokens")


def varlen_oracle_units(inp, cu, units):
    ys, ss = {}, {}
    for (s, h) in units:
        a, b = int(cu[s]), int(cu[s + 1])
        sl = lambda t: t[a:b, h][None, :, None, :].contiguous()
        s0 = None if inp.state_in is None else inp.state_in[s, h][None, None].contiguous()
        y, st = orc.prefill(sl(inp.r), sl(inp.k), sl(inp.v), sl(inp.x), inp.u[h][None].contiguous(), s0)
        ys[(s, h)], ss[(s, h)] = y[0, :, 0], st[0, 0]
    return ys, ss


@pytest.mark.parametrize("kernel", ["exact", "chunked"])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_varlen_small_full_including_empty_sequence(kernel, dtype):
    if kernel == "chunked" and dtype == "f32":
        pytest.skip("the fp32 entry points always run the exact recurrence")
    lens = [5, 0, 64, 1, 130, 77, 63, 65]
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32)
    H = 3
    inp = synth.make_varlen(cu, H, 64, dtype, seed=400, state_std=0.1)
    d = inp.to(DEV)
    gf.set_kernel(KERNELS[kernel])
    canary = 12345.0
    y = torch.full_like(d.r, canary)
    y, s = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, max(lens), d.state_in, y=y)
    gf.last_device_status()
    y_ref, s_ref = orc.prefill_varlen(inp.r, inp.k, inp.v, inp.x, inp.u, cu, inp.state_in)
    check(y, s, y_ref, s_ref, TOL[inp.r.dtype], f"varlen {kernel} {dtype}")
    # per sequence as well, so a short sequence cannot hide behind a long one
    for i in range(len(lens)):
        a, b = int(cu[i]), int(cu[i + 1])
        if b > a:
            check(y[a:b], s[i], y_ref[a:b], s_ref[i], TOL[inp.r.dtype], f"varlen seq {i}")
    assert torch.equal(s[1].cpu(), inp.state_in[1])                 # empty sequence: state passes through


@pytest.mark.parametrize("lens,H,x_hi", [([3000, 1100], 4, -1.0), ([517, 0, 2600, 64], 3, -1.0), ([1500, 2304], 2, 2.5),
                                         ([4096], 8, -1.0)])
def test_varlen_sequence_split_matches_oracle_and_unsplit_call(lens, H, x_hi):
    """Packed call with few (sequence, head) units: sequences are cut by max_seqlen, so the shorter ones
    own empty segments (identity summaries) and the last segment of each still writes the final state."""
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32)
    assert gf.workspace_bytes(len(lens), max(lens), H, 64) > 0, "this shape is expected to split"
    inp = synth.make_varlen(cu, H, 64, "bf16", seed=4400 + H, state_std=0.1, x_lo=-6.0 if x_hi < 0 else -1.0, x_hi=x_hi)
    d = inp.to(DEV)
    gf.set_kernel(gf.KERNEL_CHUNKED)
    before = gf.launch_count()
    y, s = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, max(lens), d.state_in)
    assert gf.launch_count() - before == 2
    y1, s1 = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, max(lens), d.state_in, split=False)
    assert gf.launch_count() - before == 3
    gf.last_device_status()
    y_ref, s_ref = orc.prefill_varlen(inp.r, inp.k, inp.v, inp.x, inp.u, cu, inp.state_in)
    check(y, s, y_ref, s_ref, 5e-3, "packed split")
    check(y1, s1, y_ref, s_ref, 5e-3, "packed unsplit")
    for i in range(len(lens)):
        a, b = int(cu[i]), int(cu[i + 1])
        if b > a:
            check(y[a:b], s[i], y_ref[a:b], s_ref[i], 5e-3, f"packed split seq {i}")
        else:
            assert torch.equal(s[i].cpu(), inp.state_in[i])
    assert orc.rel_l2(s.cpu().numpy(), s1.cpu().numpy()) < 1e-3


def test_cfg4_varlen_serving_then_decode_steps_every_unit():
    """Batched serving: the packed prefill of 64 sequences x 32 heads and the 256 decode steps that follow, all 2048
    (sequence, head) units against the oracle, per tensor, per unit and per token."""
    c = synth.CONFIGS["cfg4"]
    S, H = c["S"], c["H"]
    cu = synth.make_lengths(S, c["len_min"], c["len_max"], seed=4000)
    inp = synth.make_varlen(cu, H, 64, "bf16", seed=4001, device=DEV, state_std=c["state_std"])
    lens = (cu[1:] - cu[:-1])
    gf.set_kernel(gf.KERNEL_AUTO)
    y, state = gf.prefill_varlen(inp.r, inp.k, inp.v, inp.x, inp.u, inp.cu_seqlens, int(lens.max()), inp.state_in)
    gf.last_device_status()
    cpu = inp.to("cpu")
    y_ref, s_ref = orc.prefill_varlen(cpu.r, cpu.k, cpu.v, cpu.x, cpu.u, cu, cpu.state_in)
    check(y, state, y_ref, s_ref, 5e-3, "cfg4 prefill")
    yn, sn = y.float().cpu().numpy(), state.cpu().numpy()
    worst = [0.0, 0.0, 0.0]
    for i in range(S):
        a, b = int(cu[i]), int(cu[i + 1])
        w = check_units(yn[None, a:b], sn[i:i + 1], y_ref[None, a:b], s_ref[i:i + 1], f"cfg4 prefill sequence {i} ({b - a} tokens)")
        worst = [max(p, q) for p, q in zip(worst, w[2:])]
    print("cfg4 prefill: worst unit y / state / token", worst)
    # 256 decode steps per sequence, one batched call per step, state updated in place; the oracle continues from
    # ITS prefill state (rounded to fp32), so the comparison covers the whole serving sequence
    nstep = c["decode_steps"]
    dec = synth.make_dense(S, nstep, H, 64, "bf16", seed=4002, device=DEV)
    y_steps = []
    for t in range(nstep):
        yt, state = gf.step(dec.r[:, t].contiguous(), dec.k[:, t].contiguous(), dec.v[:, t].contiguous(),
                            dec.x[:, t].contiguous(), inp.u, state)
        y_steps.append(yt)
    gf.last_device_status()
    y_dec = torch.stack(y_steps, 1)                                  # [S, nstep, H, N]
    dcpu = dec.to("cpu")
    yd_ref, sd_ref = orc.prefill(dcpu.r, dcpu.k, dcpu.v, dcpu.x, cpu.u, s_ref.astype(np.float32))
    print("cfg4 decode", check_units(y_dec, state, yd_ref, sd_ref, "cfg4 decode steps"))


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_step_matches_oracle_and_prefill_of_length_one(dtype):
    B, H = 5, 7
    inp = synth.make_step(B, H, 64, dtype, seed=500)
    d = inp.to(DEV)
    s_in = d.state_in.clone()
    y, s = gf.step(d.r, d.k, d.v, d.x, d.u, s_in)                    # in place
    assert s.data_ptr() == s_in.data_ptr()
    y_ref, s_ref = orc.step(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    check(y, s, y_ref, s_ref, TOL[inp.r.dtype], "step")
    gf.set_kernel(gf.KERNEL_EXACT)
    y1, s1 = gf.prefill(d.r[:, None].contiguous(), d.k[:, None].contiguous(), d.v[:, None].contiguous(),
                        d.x[:, None].contiguous(), d.u, d.state_in)
    check(y1[:, 0], s1, y_ref, s_ref, TOL[inp.r.dtype], "prefill T=1")


def test_bound_step_loop_matches_oracle():
    """The pre-marshalled decode step over reused buffers (refreshed in place every token)."""
    B, H, T = 3, 4, 12
    inp = synth.make_dense(B, T, H, 64, "bf16", seed=650, state_std=0.1)
    d = inp.to(DEV)
    r, k, v, x = (torch.empty((B, H, 64), device=DEV, dtype=torch.bfloat16) for _ in range(4))
    state = d.state_in.clone()
    call, y = gf.bind_step(r, k, v, x, d.u, state)
    ys = []
    for t in range(T):
        r.copy_(d.r[:, t]); k.copy_(d.k[:, t]); v.copy_(d.v[:, t]); x.copy_(d.x[:, t])
        call()
        ys.append(y.clone())
    gf.last_device_status()
    y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    check(torch.stack(ys, 1), state, y_ref, s_ref, 5e-3, "bound step loop")


def test_prefill_equals_chain_of_steps():
    B, T, H = 2, 40, 2
    inp = synth.make_dense(B, T, H, 64, "f32", seed=600, state_std=0.1)
    d = inp.to(DEV)
    y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    st = d.state_in.clone()
    ys = []
    for t in range(T):
        yt, st = gf.step(d.r[:, t].contiguous(), d.k[:, t].contiguous(), d.v[:, t].contiguous(),
                         d.x[:, t].contiguous(), d.u, st)
        ys.append(yt)
    assert orc.rel_l2(torch.stack(ys, 1).cpu().numpy(), y.cpu().numpy()) < 1e-5
    assert orc.rel_l2(st.cpu().numpy(), s.cpu().numpy()) < 1e-5


@pytest.mark.parametrize("kernel", ["exact", "chunked"])
def test_state_aliasing_null_state_and_determinism(kernel):
    inp = synth.make_dense(2, 300, 4, 64, "bf16", seed=700, state_std=0.1)
    d = inp.to(DEV)
    gf.set_kernel(KERNELS[kernel])
    y1, s1 = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    inplace = d.state_in.clone()
    y2, s2 = gf.prefill(d.r, d.k, d.v, d.x, d.u, inplace, state_out=inplace)
    assert torch.equal(y1, y2) and torch.equal(s1, s2)               # aliasing + bitwise repeatability
    y3, s3 = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in, want_state=False)
    assert s3 is None and torch.equal(y1, y3)
    y4, s4 = gf.prefill(d.r, d.k, d.v, d.x, d.u, None)
    y5, s5 = gf.prefill(d.r, d.k, d.v, d.x, d.u, torch.zeros_like(d.state_in))
    assert torch.equal(y4, y5) and torch.equal(s4, s5)               # NULL state_in == zero state
    gf.last_device_status()


@pytest.mark.parametrize("kernel", ["exact", "chunked", "auto"])
@pytest.mark.parametrize("case", ["w_one", "w_zero_ish", "fast_decay", "mixed_extreme"])
def test_extreme_decay_logits(kernel, case):
    """x = -inf (w = 1), large x (w -> 0) and strongly decaying channels must stay finite and
    within tolerance: no exp overflow / underflow artefacts in the chunked factorisation."""
    B, T, H = 1, 200, 2
    inp = synth.make_dense(B, T, H, 64, "bf16", seed=800, state_std=0.1)
    g = torch.Generator().manual_seed(801)
    if case == "w_one":
        inp.x = torch.full_like(inp.x, float("-inf"))
    elif case == "w_zero_ish":
        inp.x = torch.full_like(inp.x, 10.0)
    elif case == "fast_decay":
        inp.x = (torch.rand(inp.x.shape, generator=g) * 4 - 1).bfloat16()          # U(-1, 3)
    else:
        inp.x = (torch.rand(inp.x.shape, generator=g) * 16 - 8).bfloat16()         # U(-8, 8)
        inp.x[:, ::7, :, ::5] = float("-inf")
    y, s = run_dense(inp, kernel)
    y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    assert torch.isfinite(y.float()).all() and torch.isfinite(s).all()
    check(y, s, y_ref, s_ref, 5e-3, f"{case} {kernel}")


def test_empty_time_axis_passes_state_through():
    H = 2
    u = torch.zeros((H, 64), device=DEV)
    e = torch.empty((3, 0, H, 64), device=DEV, dtype=torch.bfloat16)
    s_in = torch.randn((3, H, 64, 64), device=DEV)
    y, s = gf.prefill(e, e, e, e, u, s_in, y=torch.empty_like(e))
    assert torch.equal(s, s_in)
    y, s = gf.prefill(e, e, e, e, u, None, y=torch.empty_like(e))
    assert torch.count_nonzero(s) == 0


def test_host_buffer_entry_point():
    B, T, H = 2, 192, 3
    inp = synth.make_dense(B, T, H, 64, "bf16", seed=900, state_std=0.1)
    pin = lambda t: t.pin_memory()
    r, k, v, x, u, s0 = (pin(t) for t in (inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in))
    y = torch.empty_like(inp.r).pin_memory()
    s_out = torch.empty_like(inp.state_in).pin_memory()
    ws = torch.empty(gf.host_workspace_bytes(B, T, H, 64), dtype=torch.uint8, device=DEV)
    gf.prefill_host(r, k, v, x, u, s0, s_out, y, ws)
    gf.last_device_status()
    y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    check(y, s_out, y_ref, s_ref, 5e-3, "host entry point")


def test_calls_from_two_host_threads_on_their_own_streams():
    """The library keeps no per-call host state: two threads, each with its own stream and buffers, call the
    prefill and the decode step at the same time (shapes that do not split, so no shared workspace)."""
    import threading
    cases = [synth.make_dense(5, 200 + 70 * i, 16, 64, "bf16", seed=9100 + i, state_std=0.1) for i in range(2)]
    assert gf.workspace_bytes(5, 270, 16, 64) == 0
    results, errors = [None, None], []

    def work(i):
        try:
            torch.cuda.set_device(0)
            st = torch.cuda.Stream()
            d = cases[i].to(DEV)
            with torch.cuda.stream(st):
                for _ in range(20):
                    y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in, stream=st)
                st.synchronize()
            results[i] = (y, s)
        except Exception as e:                      # surfaced below, in the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    gf.last_device_status()
    for i, inp in enumerate(cases):
        y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
        check(results[i][0], results[i][1], y_ref, s_ref, 5e-3, f"thread {i}")


# ---- more units than SMs: one CTA per SM walks a stream of units (persistent launch)

@pytest.mark.parametrize("B,T,H,x_hi", [(40, 200, 5, -1.0), (19, 64, 16, -1.0), (33, 130, 10, 2.5), (400, 1, 1, -1.0),
                                          (7, 700, 32, -1.0)])
def test_dense_call_with_more_units_than_sms_matches_oracle(B, T, H, x_hi):
    """Several units per CTA, unit boundaries at every alignment of the ring and the double buffers (T = 64: one
    chunk per unit; T = 1: one token), strong decays that take the token-by-token path inside the stream."""
    inp = synth.make_dense(B, T, H, 64, "bf16", seed=7000 + B, state_std=0.1, x_lo=-6.0 if x_hi < 0 else -1.0, x_hi=x_hi)
    d = inp.to(DEV)
    gf.set_kernel(gf.KERNEL_CHUNKED)
    before = gf.launch_count()
    y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    assert gf.launch_count() - before == 1
    y2, s2 = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    gf.last_device_status()
    assert torch.equal(y, y2) and torch.equal(s, s2)
    y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    check(y, s, y_ref, s_ref, 5e-3, f"persistent dense B{B} T{T} H{H}")
    # every unit on its own: a unit that got another unit's state or bonus vector would show here
    yn, sn = y.float().cpu().numpy(), s.cpu().numpy()
    for b in range(0, B, max(1, B // 7)):
        for h in range(H):
            assert orc.rel_l2(yn[b, :, h], y_ref[b, :, h]) <= 6e-3, (b, h)
            assert orc.rel_l2(sn[b, h], s_ref[b, h]) <= 6e-3, (b, h)


def test_packed_call_with_more_units_than_sms_draws_units_dynamically():
    """Packed, 60 sequences x 4 heads with lengths from 0 to 300 (empty sequences, single tokens, ragged tails):
    units are handed out through the counter in the workspace; with the workspace taken away the same call
    runs one CTA per unit; both match the oracle."""
    import random
    rng = random.Random(5)
    lens = [rng.choice([0, 1, 63, 64, 65, rng.randint(2, 300)]) for _ in range(60)]
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32)
    H = 4
    inp = synth.make_varlen(cu, H, 64, "bf16", seed=7100, state_std=0.1)
    d = inp.to(DEV)
    gf.set_kernel(gf.KERNEL_CHUNKED)
    assert gf.workspace_bytes(len(lens), max(lens), H, 64) > 0
    y, s = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, max(lens), d.state_in)
    y2, s2 = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, max(lens), d.state_in)
    y1, s1 = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, max(lens), d.state_in, split=False)
    gf.last_device_status()
    assert torch.equal(y, y2) and torch.equal(s, s2)
    assert torch.equal(y, y1) and torch.equal(s, s1)      # the same arithmetic per unit, whoever runs it
    y_ref, s_ref = orc.prefill_varlen(inp.r, inp.k, inp.v, inp.x, inp.u, cu, inp.state_in)
    check(y, s, y_ref, s_ref, 5e-3, "persistent packed")
    for i, n in enumerate(lens):
        a, b = int(cu[i]), int(cu[i + 1])
        if n == 0:
            assert torch.equal(s[i].cpu(), inp.state_in[i])
        else:
            check(y[a:b], s[i], y_ref[a:b], s_ref[i], 6e-3, f"persistent packed seq {i} len {n}")


def test_persistent_launch_without_states_and_in_place_state():
    B, T, H = 30, 150, 8
    inp = synth.make_dense(B, T, H, 64, "bf16", seed=7200, state_std=0.1)
    d = inp.to(DEV)
    y0, s0 = gf.prefill(d.r, d.k, d.v, d.x, d.u, None)                       # zero start state
    st = d.state_in.clone()
    y1, s1 = gf.prefill(d.r, d.k, d.v, d.x, d.u, st, state_out=st)            # state updated in place
    y2, _ = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in, want_state=False)  # no final state wanted
    gf.last_device_status()
    y_ref0, s_ref0 = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, None)
    y_ref1, s_ref1 = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    check(y0, s0, y_ref0, s_ref0, 5e-3, "zero state")
    check(y1, s1, y_ref1, s_ref1, 5e-3, "in place")
    assert torch.equal(y1, y2)


def test_random_many_unit_shapes_against_oracle():
    """Seeded sweep over calls with more units than SMs: dense and packed, lengths with every kind of tail, decay
    ranges from tame to chunks that all take the token-by-token path; every unit against the oracle."""
    import random
    rng = random.Random(20240713)
    gf.set_kernel(gf.KERNEL_CHUNKED)
    for it in range(14):
        H = rng.choice([1, 2, 3, 5, 8, 16])
        units = rng.randint(149, 900)
        x_lo, x_hi = rng.choice([(-6.0, -1.0), (-6.0, -1.0), (-3.0, 1.5), (-1.0, 2.5), (-8.0, 0.5)])
        if rng.random() < 0.5:
            S = max(1, units // H)
            lens = [rng.choice([0, 1, 63, 64, 65, 128, rng.randint(1, 330)]) for _ in range(S)]
            lens[0] = max(lens[0], 3)
            cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32)
            inp = synth.make_varlen(cu, H, 64, "bf16", seed=9100 + it, state_std=0.1, x_lo=x_lo, x_hi=x_hi)
            d = inp.to(DEV)
            y, s = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, max(lens), d.state_in)
            gf.last_device_status()
            y_ref, s_ref = orc.prefill_varlen(inp.r, inp.k, inp.v, inp.x, inp.u, cu, inp.state_in)
            yn, sn = y.float().cpu().numpy(), s.cpu().numpy()
            for i, n in enumerate(lens):
                a, b = int(cu[i]), int(cu[i + 1])
                for h in range(H):
                    if n == 0:
                        assert np.array_equal(sn[i, h], inp.state_in[i, h].numpy()), (it, i, h)
                    else:
                        assert orc.rel_l2(yn[a:b, h], y_ref[a:b, h]) <= 6e-3 and orc.rel_l2(sn[i, h], s_ref[i, h]) <= 6e-3, (it, i, h, n)
        else:
            B, T = max(1, units // H), rng.choice([1, 7, 64, 65, 128, 129, 192, rng.randint(2, 330)])
            inp = synth.make_dense(B, T, H, 64, "bf16", seed=9100 + it, state_std=0.1, x_lo=x_lo, x_hi=x_hi)
            d = inp.to(DEV)
            y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
            gf.last_device_status()
            y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
            yn, sn = y.float().cpu().numpy(), s.cpu().numpy()
            for b in range(B):
                for h in range(H):
                    assert orc.rel_l2(yn[b, :, h], y_ref[b, :, h]) <= 6e-3 and orc.rel_l2(sn[b, h], s_ref[b, h]) <= 6e-3, (it, b, h, T)


@pytest.mark.parametrize("S", [5000, 8200])
def test_packed_call_with_thousands_of_short_sequences(S):
    """Thousands of sequences of 0..3 tokens, one head: the rank kernel at its size limit (S = 5000) and the
    index-order fallback beyond it (S = 8200); every sequence against the oracle."""
    import random
    rng = random.Random(S)
    lens = [rng.randint(0, 3) for _ in range(S)]
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32)
    inp = synth.make_varlen(cu, 1, 64, "bf16", seed=7300 + S, state_std=0.1)
    d = inp.to(DEV)
    gf.set_kernel(gf.KERNEL_CHUNKED)
    y, s = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, 3, d.state_in)
    gf.last_device_status()
    y_ref, s_ref = orc.prefill_varlen(inp.r, inp.k, inp.v, inp.x, inp.u, cu, inp.state_in)
    check(y, s, y_ref, s_ref, 5e-3, f"{S} short sequences")
    sn = s.cpu().numpy()
    worst = max(orc.rel_l2(sn[i], s_ref[i]) for i in range(S))
    assert worst <= 6e-3, worst
    empty = [i for i, n in enumerate(lens) if n == 0]
    assert all(np.array_equal(sn[i], inp.state_in[i].numpy()) for i in empty[:200])


@pytest.mark.parametrize("H", [32769, 65536, 65537])
@pytest.mark.parametrize("form", ["dense", "packed", "c2", "train"])
def test_more_heads_than_15_bits(H, form):
    """A streamed launch hands the head on in the 16 upper bits of a chunk's descriptor; more heads run one CTA per unit."""
    T = 3
    i = synth.make_dense(1, T, H, 64, "bf16", seed=H, device=DEV)
    if form == "dense":
        y, _ = gf.prefill(i.r, i.k, i.v, i.x, i.u, None, want_state=False)
    elif form == "packed":
        cu = torch.tensor([0, 1, T], dtype=torch.int32, device=DEV)
        y, _ = gf.prefill_varlen(i.r[0], i.k[0], i.v[0], i.x[0], i.u, cu, 2, None, want_state=False)
        y = y[None]
    elif form == "c2":
        y, _ = gf.prefill_c2(i.r, i.k, i.v, i.x, None, None, want_state=False)
    else:
        ws = torch.empty(gf.backward_workspace_bytes(1, T, H, 64), dtype=torch.uint8, device=DEV)
        y, _ = gf.prefill_train(i.r, i.k, i.v, i.x, i.u, ws, None)
    gf.last_device_status()
    heads = torch.tensor([0, 1, 32767, 32768, H // 2, H - 2, H - 1])
    c = [t[:, :, heads.to(DEV)].contiguous().cpu() for t in (i.r, i.k, i.v, i.x)]
    u = i.u[heads.to(DEV)].cpu()
    if form == "c2":
        ref, _ = orc.prefill_c2(*c, None, None)
    elif form == "packed":
        ref = np.concatenate([orc.prefill(*(t[:, a:b].contiguous() for t in c), u, None)[0] for a, b in ((0, 1), (1, T))], axis=1)
    else:
        ref, _ = orc.prefill(*c, u, None)
    got = y[:, :, heads.to(DEV)].float().cpu().numpy()
    for n in range(len(heads)):
        assert orc.rel_l2(got[:, :, n], ref[:, :, n]) <= 2 * 2.0 ** -8, int(heads[n])      # (three tokens of one head: two bf16 roundings)
    assert torch.isfinite(y.float()).all()
