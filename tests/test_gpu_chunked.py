"""The general chunked kernels (float32 arithmetic on CUDA cores) at the edges of
their tiles: lengths around the 32-token chunk, every pair of head dimensions,
and sequence counts that select each width of the inter-chunk passes (16, 32 or 64
value columns a CTA: the widest that leaves at least 120 CTAs)."""
import numpy as np
import pytest
import torch

import oracle
from kdn_inputs import make_inputs
from kdn_gpu_util import check, to_dev

pytestmark = pytest.mark.gpu
NAMES = ("q", "k", "v", "g", "omega", "r")
GRADS = ("dq", "dk", "dv", "dg", "domega", "dr", "dS0", "dp0", "dmu")

# variant, per-channel decay, B, T, H, dk, dv
CASES = [("diag", True, 1, T, 2, 64, 64) for T in (1, 31, 32, 33, 65)]
CASES += [("iso", pc, 1, T, 2, 64, 64) for pc in (False, True) for T in (1, 33, 64)]
CASES += [(v, v == "diag", 1, 40, 3, dk, dv) for v in ("diag", "iso")
          for dk in (32, 64, 128) for dv in (32, 64, 128)]
CASES += [("diag", True, 8, 34, 15, dk, dv) for dk, dv in ((32, 64), (64, 64), (128, 128))]
CASES += [("diag", True, 4, 34, 15, 64, 64), ("iso", False, 4, 34, 16, 128, 64)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_chunked_forward_and_backward(case):
    variant, pc, B, T, H, dk, dv = case
    from paper_2609_07816_gb300 import build
    build.build()
    import paper_2609_07816_gb300 as kdn
    ins = make_inputs(variant, B, T, H, dk, dv, dtype="f32", seed=T + dk + dv, s0_std=0.1,
                      p0_range=(0.5, 2.0), per_channel_decay=pc, with_grad=True)
    d = to_dev(ins)
    x = [d[n] for n in NAMES]
    fwd, bwd = ((kdn.kdn_diag_fwd, kdn.kdn_diag_bwd) if variant == "diag"
                else (kdn.kdn_iso_fwd, kdn.kdn_iso_bwd))
    o, ST, pT = fwd(*x, d["S0"], d["p0"], chunk=32)
    rng = np.random.default_rng(7)
    dST, dpT = rng.standard_normal(ST.shape), rng.standard_normal(pT.shape)
    cu = lambda y: torch.tensor(y, dtype=torch.float32, device="cuda")
    gr = bwd(*x, d["S0"], d["p0"], d["dO"], cu(dST), cu(dpT), chunk=32)
    torch.cuda.synchronize()
    f32 = lambda y: np.float64(np.float32(y))
    ref = oracle.fwd(variant, *[ins[n] for n in NAMES], ins["S0"], ins["p0"])
    rg = oracle.bwd(variant, *[ins[n] for n in NAMES], ins["S0"], ins["p0"], ins["dO"],
                    f32(dST), f32(dpT))
    for n, y in (("o", o), ("ST", ST), ("pT", pT)):
        check(n, y, ref[n], "f32")
    for n in GRADS:
        check(n, gr[n], rg[n], "f32")
