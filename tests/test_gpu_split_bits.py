"""The two-kernel backward of the Diagonal KDN gives the one-kernel sweep's gradients bit for
bit: both multiply the same 16-bit operands in the same order, and the chunks hand on the
uncertainty cotangent that the recursion itself ends with.  The sweep is the route of a call
that also wants the state gradients."""
import numpy as np
import pytest
import torch

from kdn_gpu_util import to_dev
from kdn_inputs import round_to
from test_gpu_split import GRADS, NAMES, _case

pytestmark = pytest.mark.gpu

SIZES = [(2, 512, 6, "post", False), (2, 512, 6, "logits", True), (1, 1000, 8, "post", True),
         (2, 449, 6, "logits", False), (40, 190, 1, "post", False), (33, 191, 1, "logits", True),
         (4, 1024, 16, "post", False), (2, 1999, 16, "logits", True)]


# low: noise and uncertainty of ~1e-4, where phat k would lie among fp16's subnormal numbers
@pytest.mark.parametrize("low", [False, True])
@pytest.mark.parametrize("B,T,H,gates,slow", SIZES)
def test_two_kernels_equal_the_sweep(B, T, H, gates, slow, low):
    from paper_2609_07816_gb300 import build
    build.build()
    import paper_2609_07816_gb300 as kdn
    ins, dST, dpT = _case(B, T, H, T + B, gates, slow)
    if low:
        if gates == "logits":
            for n in ("omega", "r"):
                ins[n] = round_to(ins[n] - 9.0, "bf16")
        else:
            for n in ("omega", "r"):
                ins[n] = round_to(ins[n] * 2.0 ** -13, "bf16")
        ins["p0"] = ins["p0"] * np.float32(2.0 ** -13)
    d = to_dev(ins)
    x = [d[n] for n in NAMES]
    G = kdn.KDN_GATES_LOGITS if gates == "logits" else kdn.KDN_GATES_POST
    desc = kdn.make_desc(B, T, H, 128, 128, torch.bfloat16, out_dtype=torch.bfloat16, gates=G, r_min=0.0)
    kw = dict(out_dtype=torch.bfloat16, gates=G, r_min=0.0, workspace=kdn.alloc_workspace(desc, 0, "saved"))
    cu = lambda y: torch.tensor(y, dtype=torch.float32, device="cuda")
    _, _, _, saved = kdn.kdn_diag_fwd_save(*x, d["S0"], d["p0"], **kw)
    for end in ((cu(dST), cu(dpT)), (None, None)):
        sweep = kdn.kdn_diag_bwd_saved(*x, saved, d["dO"], *end, **kw)
        two = kdn.kdn_diag_bwd_saved(*x, saved, d["dO"], *end, want_state_grads=False, **kw)
        torch.cuda.synchronize()
        assert kdn.kdn_get_device_status(kw["workspace"]) == 0
        for n in GRADS:
            assert torch.isfinite(sweep[n]).all(), n
            assert torch.equal(sweep[n], two[n]), n
