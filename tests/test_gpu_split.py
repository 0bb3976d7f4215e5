"""The two-kernel backward of the Diagonal KDN (bf16, d = 128, bf16 gradients without state
gradients): whole chunks (scratch in the gradient buffers) and ragged lengths (scratch in
the workspace), both gate forms, a slow decay that carries the cotangents over many chunks,
against the oracle; and the one-kernel sweep that reads the same context when state
gradients are wanted, the gradients are float32, or the workspace has no room.

Gradients are compared in the 2-norm: with a slow decay or logit gates their entries are
heavy-tailed and the largest error over the RMS says little (the one-kernel sweep has
5e-2 there).  A gradient passes at most eight 16-bit operand roundings of 2^-11 each
between dO and its store, so 2^-8 relative, and 2^-9 more when stored in bf16."""
import numpy as np
import pytest
import torch

import oracle
from kdn_inputs import make_inputs, round_to
from kdn_gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu
NAMES = ("q", "k", "v", "g", "omega", "r")
GRADS = ("dq", "dk", "dv", "dg", "domega", "dr")


@pytest.fixture(scope="module")
def kdn():
    from paper_2609_07816_gb300 import build
    build.build()
    import paper_2609_07816_gb300 as m
    return m


def check(name, x, ref, bf16_store=False):
    err = np.linalg.norm(to_np(x) - ref) / np.linalg.norm(ref)
    assert err <= 2.0 ** -8 + (2.0 ** -9 if bf16_store else 0.0), f"{name}: {err:.2e}"


def _case(B, T, H, seed, gates, slow):
    ins = make_inputs("diag", B, T, H, 128, 128, dtype="bf16", seed=seed, s0_std=0.05,
                      p0_range=(0.5, 2.0), with_grad=True)
    rng = np.random.default_rng(seed)
    x = rng.normal(6.0 if slow else 2.0, 1.0, size=ins["g"].shape)
    if gates == "logits":
        ins["g"] = round_to(x, "bf16")
        ins["omega"] = round_to(rng.standard_normal(ins["omega"].shape), "bf16")
        ins["r"] = round_to(rng.standard_normal(ins["r"].shape), "bf16")
    elif slow:
        ins["g"] = round_to(-np.logaddexp(0.0, -x), "bf16")
    return ins, rng.standard_normal((B, H, 128, 128)) * 0.05, rng.standard_normal((B, H, 128)) * 0.05


@pytest.mark.parametrize("out", ["f32", "bf16"])
@pytest.mark.parametrize("B,T,H,gates,slow", [
    (2, 512, 6, "post", False), (2, 512, 6, "logits", True), (1, 1000, 8, "post", True),
    (2, 449, 6, "logits", False), (40, 190, 1, "post", False), (96, 64, 1, "post", False),
    (97, 1, 1, "logits", False), (33, 191, 1, "post", True)])
def test_split_backward(kdn, B, T, H, gates, slow, out):
    ins, dST, dpT = _case(B, T, H, T + B, gates, slow)
    d = to_dev(ins)
    x = [d[n] for n in NAMES]
    dt = torch.float32 if out == "f32" else torch.bfloat16
    G = kdn.KDN_GATES_LOGITS if gates == "logits" else kdn.KDN_GATES_POST
    desc = kdn.make_desc(B, T, H, 128, 128, torch.bfloat16, out_dtype=dt, gates=G)
    kw = dict(out_dtype=dt, gates=G, workspace=kdn.alloc_workspace(desc, 0))
    o, _, _, saved = kdn.kdn_diag_fwd_save(*x, d["S0"], d["p0"], **kw)
    cu = lambda y: torch.tensor(y, dtype=torch.float32, device="cuda")
    gr = kdn.kdn_diag_bwd_saved(*x, saved, d["dO"], cu(dST), cu(dpT), **kw)
    plain = kdn.kdn_diag_bwd_saved(*x, saved, d["dO"], cu(dST), cu(dpT), want_state_grads=False, **kw)
    again = kdn.kdn_diag_bwd_saved(*x, saved, d["dO"], cu(dST), cu(dpT), want_state_grads=False, **kw)
    full = kdn.kdn_diag_bwd(*x, d["S0"], d["p0"], d["dO"], cu(dST), cu(dpT), out_dtype=dt, gates=G,
                            want_state_grads=False)
    torch.cuda.synchronize()
    assert kdn.kdn_get_device_status(kw["workspace"]) == 0
    f32 = lambda y: np.float64(np.float32(y))
    rg = oracle.bwd("diag", *[ins[n] for n in NAMES], ins["S0"], ins["p0"], ins["dO"], f32(dST),
                    f32(dpT), gates=gates, r_min=kdn.R_MIN_DEFAULT)
    for n in GRADS:
        check(n, plain[n], rg[n], out == "bf16")
        check(n, gr[n], rg[n], out == "bf16")
        # the context is only read, the result does not depend on who runs first
        assert torch.equal(plain[n], again[n]) and torch.equal(plain[n], full[n]), n
    for n in ("dS0", "dp0", "dmu"):
        check(n, gr[n], rg[n])
    # the routes round differently; one chunk of each sequence is the sweep's
    assert torch.equal(plain["dk"], gr["dk"]) == (out == "f32" or T <= 64)


@pytest.mark.parametrize("first,then", [("f32", "bf16"), ("bf16", "f32")])
def test_context_serves_either_gradient_type(kdn, first, then):
    """The context does not depend on the type that o was stored in."""
    ins, dST, dpT = _case(2, 449, 6, 5, "post", False)
    d = to_dev(ins)
    x = [d[n] for n in NAMES]
    dt = {"f32": torch.float32, "bf16": torch.bfloat16}
    _, _, _, saved = kdn.kdn_diag_fwd_save(*x, d["S0"], d["p0"], out_dtype=dt[first])
    gr = kdn.kdn_diag_bwd_saved(*x, saved, d["dO"], want_state_grads=False, out_dtype=dt[then])
    rg = oracle.bwd("diag", *[ins[n] for n in NAMES], ins["S0"], ins["p0"], ins["dO"])
    for n in GRADS:
        check(n, gr[n], rg[n], then == "bf16")


@pytest.mark.parametrize("out", ["f32", "bf16"])
@pytest.mark.parametrize("B,T,H,gates,slow,fast", [
    (1, 824, 16, "post", False, 0), (2, 1985, 14, "logits", True, 0), (1, 1537, 5, "post", False, 9.0),
    (2, 1100, 12, "logits", False, 9.0), (1, 700, 10, "post", True, 0), (2, 1000, 16, "post", False, 0)])
def test_flow_forward_equals_the_one(kdn, B, T, H, gates, slow, fast, out):
    """The gain, the chunk part and the memory part on CTAs of their own run the same arithmetic: the
    outputs are those of the one-kernel forward (a workspace without room) bit for bit, also
    where a chunk's decay leaves the referenced range (fast: log alpha of -9)."""
    ins, _, _ = _case(B, T, H, T + B, gates, slow)
    if fast:  # some channels decay by e^-9 a token (logits: log sigmoid(-9))
        ins["g"][:, T // 2:, :, ::5] = -fast
    d = to_dev(ins)
    x = [d[n] for n in NAMES]
    dt = torch.float32 if out == "f32" else torch.bfloat16
    G = kdn.KDN_GATES_LOGITS if gates == "logits" else kdn.KDN_GATES_POST
    desc = kdn.make_desc(B, T, H, 128, 128, torch.bfloat16, out_dtype=dt, gates=G)
    assert kdn.workspace_bytes(desc, 0) >= B * H * ((T + 63) // 64) * 66560  # its records
    kw = dict(out_dtype=dt, gates=G)
    for state in ((d["S0"], d["p0"]), (None, None)):
        ws = kdn.alloc_workspace(desc, 0)
        three = kdn.kdn_diag_fwd(*x, *state, workspace=ws, **kw)
        one = kdn.kdn_diag_fwd(*x, *state, workspace=torch.empty(256, dtype=torch.uint8, device="cuda"), **kw)
        saving = kdn.kdn_diag_fwd_save(*x, *state, **kw)
        torch.cuda.synchronize()
        assert kdn.kdn_get_device_status(ws) == 0
        for u, v, w in zip(three, one, saving):
            assert torch.equal(u, v)
            assert fast or torch.equal(v, w)  # (the context keeps the referenced form)


def test_ragged_without_scratch_runs_the_sweep(kdn):
    """A workspace that holds only the status word: the one-kernel sweep reads the same context."""
    ins, dST, dpT = _case(2, 449, 6, 3, "post", True)
    d = to_dev(ins)
    x = [d[n] for n in NAMES]
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    _, _, _, saved = kdn.kdn_diag_fwd_save(*x, d["S0"], d["p0"], workspace=ws)
    gr = kdn.kdn_diag_bwd_saved(*x, saved, d["dO"], workspace=ws, out_dtype=torch.bfloat16, want_state_grads=False)
    torch.cuda.synchronize()
    assert kdn.kdn_get_device_status(ws) == 0
    rg = oracle.bwd("diag", *[ins[n] for n in NAMES], ins["S0"], ins["p0"], ins["dO"])
    for n in GRADS:
        check(n, gr[n], rg[n], True)
