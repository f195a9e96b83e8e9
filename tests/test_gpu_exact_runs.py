"""The token-by-token fp32 kernel's split of the tokens into runs, blocks and clusters (csrc/wkv6_exact.cuh), against the fp64
oracle: every launch form at lengths around its blocks, and decays whose products over a run leave fp32's range."""
import numpy as np
import pytest
import torch

import paper_2407_12077_b200 as gf
from oracle import wkv6_oracle as orc
from paper_2407_12077_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TOL = 1e-4                      # the contract's for fp32 inputs


@pytest.fixture(autouse=True)
def _status():
    yield
    gf.set_kernel(gf.KERNEL_AUTO)
    gf.last_device_status()


# heads on both sides of each rule of launch_exact (148 SMs), lengths around the blocks and rounds of the form taken
@pytest.mark.parametrize("H,T", [(4, 1), (4, 4), (4, 5), (60, 3), (4, 64), (4, 65), (4, 255), (4, 257), (4, 300), (8, 96), (8, 97), (8, 513), (12, 384), (12, 385),
                                 (20, 385), (32, 390), (36, 130), (40, 127), (40, 128), (40, 193), (60, 65), (80, 130)])
def test_launch_forms(H, T):
    inp = synth.make_dense(1, T, H, 64, "f32", seed=1000 * H + T, state_std=0.1)
    d = inp.to(DEV)
    y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    st = d.state_in.clone()
    y2, _ = gf.prefill(d.r, d.k, d.v, d.x, d.u, st, state_out=st)             # the state updated in place
    assert torch.equal(y, y2) and torch.equal(s, st)
    y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    assert orc.rel_l2(y.cpu().numpy(), y_ref) <= TOL and orc.rel_l2(s.cpu().numpy(), s_ref) <= TOL


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("H", [1, 6, 20])
def test_packed_lengths(H, dtype):
    lens = [0, 1, 63, 500, 0, 130, 64, 257]
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32)
    if H == 20:
        cu = cu[:3]                                                          # (forty units)
    inp = synth.make_varlen(cu, H, 64, dtype, seed=77 + H, state_std=0.1)
    d = inp.to(DEV)
    gf.set_kernel(gf.KERNEL_EXACT)
    y, s = gf.prefill_varlen(d.r, d.k, d.v, d.x, d.u, d.cu_seqlens, int((cu[1:] - cu[:-1]).max()), d.state_in)
    y_ref, s_ref = orc.prefill_varlen(inp.r, inp.k, inp.v, inp.x, inp.u, inp.cu_seqlens, inp.state_in)
    tol = TOL if dtype == "f32" else 5e-3
    assert orc.rel_l2(y.float().cpu().numpy(), y_ref) <= tol and orc.rel_l2(s.cpu().numpy(), s_ref) <= TOL


@pytest.mark.parametrize("H,T", [(4, 256), (4, 600), (8, 256), (12, 400), (20, 400), (40, 200), (60, 70)])
@pytest.mark.parametrize("x", [0.2, 0.5, 2.4])
def test_products_of_decays_that_underflow(H, T, x):
    """A large start state that nothing is added to: what the decays have left of it is right to the last row that fp32 holds,
    also where their product over a run or a block is below fp32's range.  2^-24 per multiplication, T of them at most."""
    inp = synth.make_dense(1, T, H, 64, "f32", seed=5, state_std=1e20)
    inp.k.zero_()
    inp.x.fill_(x)
    inp.x[:, :, :, ::3] = -4.0                                               # (a third of the channels decays slowly)
    inp.r[:, :, :, ::3] = 0.0                                                # ... and is not looked at in y
    d = inp.to(DEV)
    y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    y_ref, s_ref = orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in)
    y, y_ref = y.double().cpu().numpy(), np.asarray(y_ref)
    scale = np.sqrt((y_ref ** 2).mean(-1))
    rows = scale > 1e-30                                                     # (subnormal states before that)
    err = np.sqrt(((y - y_ref) ** 2).mean(-1))[rows] / scale[rows]
    assert rows[0, :5].all() and err.max() <= 1e-4
    assert orc.rel_l2(s.cpu().numpy()[:, :, ::3], np.asarray(s_ref)[:, :, ::3]) <= TOL


def test_values_that_are_not_finite_stay_where_they_are():
    """NaN and infinity in single channels, and decays of exactly zero and one: the same elements are non-finite as in the oracle."""
    inp = synth.make_dense(1, 300, 4, 64, "f32", seed=9, state_std=0.1)
    inp.x[0, 70, 0, 3] = float("nan")
    inp.k[0, 200, 1, 5] = float("inf")
    inp.v[0, 130, 2, 7] = float("nan")
    inp.x[0, 40:60, 3, :] = float("inf")                                     # w = 0: forgets all, finitely
    inp.x[0, 100:200, 3, 8:16] = float("-inf")                               # w = 1
    d = inp.to(DEV)
    y, s = gf.prefill(d.r, d.k, d.v, d.x, d.u, d.state_in)
    y_ref, s_ref = (np.asarray(a) for a in orc.prefill(inp.r, inp.k, inp.v, inp.x, inp.u, inp.state_in))
    y, s = y.double().cpu().numpy(), s.double().cpu().numpy()
    assert (np.isfinite(y) == np.isfinite(y_ref)).all() and (np.isfinite(s) == np.isfinite(s_ref)).all()
    ok = np.isfinite(y_ref)
    assert np.linalg.norm(y[ok] - y_ref[ok]) <= TOL * np.linalg.norm(y_ref[ok])
