"""Kernels that may be scheduled before the one ahead of them in the stream has finished: calls enqueued back to back, each
reading what the one before wrote, give bit for bit what they give with a synchronisation after every call."""
import pytest
import torch

import paper_2407_12077_b200 as gf
from paper_2407_12077_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def chain(calls, inp, sync):
    v, out = inp, []
    for call in calls:
        v = call(v)
        out.append(v)
        if sync:
            torch.cuda.synchronize()
    torch.cuda.synchronize()
    gf.last_device_status()
    return out


# one short unit; fewer units than SMs; a stream of units per SM; split into segments (short and long); balanced
@pytest.mark.parametrize("B,T,H", [(1, 5, 1), (3, 333, 4), (60, 40, 8), (1, 2500, 4), (1, 13000, 4), (5, 500, 32)])
@pytest.mark.parametrize("c2", [False, True])
def test_dense_prefills_and_norms_in_a_chain(B, T, H, c2):
    d = synth.make_dense(B, T, H, 64, "bf16", seed=5, device=DEV, state_std=0.1)
    gamma = torch.full((64 * H,), 0.5, device=DEV)

    def prefill(v):
        f = lambda: gf.prefill_c2(d.r, d.k, v, d.x, None, d.state_in) if c2 else gf.prefill(d.r, d.k, v, d.x, d.u, d.state_in)
        return f()[0]

    def norm(y):
        return gf.layernorm_heads(y, gamma, None, 1e-5)

    calls = [prefill, norm, prefill, prefill, norm, norm, prefill, norm]
    for a, b in zip(chain(calls, d.v, False), chain(calls, d.v, True)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("S,H", [(5, 4), (40, 8)])
def test_packed_prefills_whose_lengths_come_from_the_kernel_before(S, H):
    """cu_seqlens written by the operation ahead of the call (and overwritten after it)."""
    g = torch.Generator().manual_seed(3)
    lens = torch.randint(1, 300, (S,), generator=g)
    cu = torch.cat([torch.zeros(1, dtype=torch.int64), lens.cumsum(0)]).to(torch.int32)
    d = synth.make_varlen(cu, H, 64, "bf16", seed=7, device=DEV, state_std=0.1)
    cu_d, hold = d.cu_seqlens.clone(), d.cu_seqlens.clone()
    mx = int(lens.max())

    def prefill(v):
        hold.copy_(cu_d)
        y = gf.prefill_varlen(d.r, d.k, v, d.x, d.u, hold, mx, d.state_in)[0]
        hold.zero_()
        return y

    calls = [prefill] * 6
    for a, b in zip(chain(calls, d.v, False), chain(calls, d.v, True)):
        assert torch.equal(a, b)


def test_decay_logits_into_the_prefill():
    B, T, H = 2, 700, 4
    d = synth.make_dense(B, T, H, 64, "bf16", seed=9, device=DEV)
    w = synth.make_decay_lora(64 * H, 32, 64, seed=2, device=DEV)

    def step(v):
        x = gf.decay_logit(v.view(B, T, 64 * H), w["mu_x"], w["A_d"], w["B_d"], w["lambda_d"], w["A_w"], w["B_w"], w["lambda_w"])
        return gf.prefill_c2(d.r, d.k, v, x.view(B, T, H, 64))[0]

    calls = [step] * 6
    for a, b in zip(chain(calls, d.v, False), chain(calls, d.v, True)):
        assert torch.equal(a, b)
