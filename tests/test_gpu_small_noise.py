"""The general chunked kernels where the noises are far apart: observation noise down to 1e-30
(the header asks for r > 0 only), process noise up to 1e4 beside a decay of e^-83 a chunk,
and lengths of more than eight chunks, whose scans run over several blocks."""
import numpy as np
import pytest
import torch

import oracle
from kdn_gpu_util import check, to_dev
from kdn_inputs import make_inputs, round_to

pytestmark = pytest.mark.gpu
NAMES = ("q", "k", "v", "g", "omega", "r")


def _call(variant, ins, grads, **kw):
    from paper_2609_07816_gb300 import build
    build.build()
    import paper_2609_07816_gb300 as kdn
    d = to_dev(ins)
    x = [d[n] for n in NAMES]
    fwd, bwd = ((kdn.kdn_diag_fwd, kdn.kdn_diag_bwd) if variant == "diag"
                else (kdn.kdn_iso_fwd, kdn.kdn_iso_bwd))
    out = dict(zip(("o", "ST", "pT"), fwd(*x, d["S0"], d["p0"], **kw)))
    if grads:
        out.update(bwd(*x, d["S0"], d["p0"], d["dO"], **kw))
    return out


def _run(variant, ins, grads):
    out = _call(variant, ins, grads)
    args = [ins[n] for n in NAMES] + [ins["S0"], ins["p0"]]
    ref = oracle.fwd(variant, *args)
    if grads:
        ref.update(oracle.bwd(variant, *args, ins["dO"]))
    for n, y in out.items():
        check(n, y, ref[n], "f32")


def _ins(variant, T, d, dv=None, B=2, H=3, per_channel=True):
    return make_inputs(variant, B, T, H, d, dv or d, dtype="f32", seed=T + d, s0_std=0.1,
                       p0_range=(0.5, 2.0), per_channel_decay=per_channel, with_grad=True)


@pytest.mark.parametrize("one_hot", [False, True])
@pytest.mark.parametrize("r,w", [(1e-6, 100.0), (1e-8, 1.0), (1e-10, 1.0), (1e-20, 1.0), (1e-30, 1.0)])
@pytest.mark.parametrize("variant,d", [("diag", 32), ("diag", 64), ("diag", 128), ("iso", 64)])
def test_small_observation_noise(variant, d, r, w, one_hot):
    ins = _ins(variant, 300, d, per_channel=variant == "diag")
    rng = np.random.default_rng(1)
    ins["r"] = round_to(r * rng.uniform(0.5, 2.0, ins["r"].shape), "f32")
    ins["omega"] = round_to(w * ins["omega"], "f32")
    if one_hot:
        k = np.zeros_like(ins["k"])
        np.put_along_axis(k, rng.integers(0, d, k.shape[:-1] + (1,)), 1.0, -1)
        ins["k"] = k
    # (gradients: finite.  The part of domega and dp0 that is left where k is one-hot is the
    # difference of numbers 1e6 times as large, in any order of operations)
    _run(variant, ins, False)
    if r >= 1e-10:
        assert all(torch.isfinite(t).all() for t in _call(variant, ins, True).values())


def test_small_noise_from_logits():
    """softplus(-24) rounds to an observation noise of 0: everything stays finite."""
    ins = _ins("diag", 300, 64)
    rng = np.random.default_rng(2)
    ins["g"] = round_to(rng.normal(2.0, 1.0, ins["g"].shape), "f32")
    ins["omega"] = round_to(rng.standard_normal(ins["omega"].shape), "f32")
    ins["r"] = round_to(rng.normal(-24.0, 1.0, ins["r"].shape), "f32")
    out = _call("diag", ins, False, gates=1, r_min=0.0)
    assert all(torch.isfinite(t).all() for t in out.values())


@pytest.mark.parametrize("d", [32, 64, 128])
def test_strong_decay_and_large_process_noise(d):
    """phat k / gamma alone is beyond float32 at the end of a 32-token chunk."""
    ins = _ins("diag", 100, d)
    ins["g"][..., ::3] = np.float32(-83.0 / 32)
    ins["omega"] = round_to(1e4 * ins["omega"], "f32")
    _run("diag", ins, True)


@pytest.mark.parametrize("variant,pc,T,d,dv", [("diag", True, 300, 64, 64), ("diag", True, 577, 128, 32),
                                               ("iso", False, 300, 64, 64), ("iso", True, 777, 32, 128)])
def test_scans_over_several_blocks(variant, pc, T, d, dv):
    _run(variant, _ins(variant, T, d, dv, per_channel=pc), True)
