"""The context that k_wy_flow leaves (its hand-over lies in the same records), read by beta_eff; and
two of its calls in flight at once, each with a workspace of its own."""
import numpy as np
import pytest
import torch

import oracle
from kdn_gpu_util import check, to_dev, to_np
from test_gpu_split import GRADS, NAMES, _case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kdn():
    from paper_2609_07816_gb300 import build
    build.build()
    import paper_2609_07816_gb300 as m
    return m


@pytest.mark.parametrize("gates", ["post", "logits"])
def test_beta_eff_beyond_96_chunks(kdn, gates):
    ins, _, _ = _case(1, 897, 8, 11, gates, False)  # 15 chunks of 8 sequences, one token in the last
    d = to_dev(ins)
    kw = dict(gates=kdn.KDN_GATES_LOGITS if gates == "logits" else kdn.KDN_GATES_POST, r_min=0.01)
    _, _, _, saved = kdn.kdn_diag_fwd_save(*[d[n] for n in NAMES], d["S0"], d["p0"], **kw)
    be = kdn.kdn_diag_beta_eff(d["k"], d["v"], d["g"], d["r"], saved, **kw)
    torch.cuda.synchronize()
    ref = oracle.fwd("diag", *[ins[n] for n in NAMES], ins["S0"], ins["p0"], trace=True, gates=gates, r_min=0.01)
    check("beta_eff", be, np.sum(ins["k"].astype(np.float64) * ref["kappa"], axis=-1), "bf16")
    assert np.all(to_np(be) >= 0) and np.all(to_np(be) < 1)


def test_two_streams_with_a_workspace_each(kdn):
    bf = torch.bfloat16
    sides, jobs = [torch.cuda.Stream() for _ in range(3)], []
    for i, (B, T, H) in enumerate(((1, 897, 8), (2, 1999, 16), (1, 2047, 14))):
        d = to_dev(_case(B, T, H, i, "post", False)[0])
        x = [d[n] for n in NAMES]
        desc = kdn.make_desc(B, T, H, 128, 128, bf, out_dtype=bf)
        ws = kdn.alloc_workspace(desc, 0), kdn.alloc_workspace(desc, 0, "saved")
        e = lambda t: torch.empty_like(t)
        bufs = dict(o=e(x[2]), o2=e(x[2]), saved=torch.empty(kdn.saved_bytes(desc), dtype=torch.uint8, device="cuda"),
                    **{n: e(t) for n, t in zip(GRADS, x)})

        def run(stream, x=x, d=d, ws=ws, bufs=bufs):
            kw = dict(out_dtype=bf, stream=stream)
            kdn.kdn_diag_fwd(*x, d["S0"], d["p0"], o=bufs["o"], want_state=False, workspace=ws[0], **kw)
            kdn.kdn_diag_fwd_save(*x, d["S0"], d["p0"], o=bufs["o2"], want_state=False, saved=bufs["saved"],
                                  workspace=ws[0], **kw)
            kdn.kdn_diag_bwd_saved(*x, bufs["saved"], d["dO"], grads={n: bufs[n] for n in GRADS},
                                   want_state_grads=False, workspace=ws[1], **kw)

        run(None)
        torch.cuda.synchronize()
        outs = {n: t for n, t in bufs.items() if n != "saved"}
        jobs.append((run, outs, {n: t.clone() for n, t in outs.items()}, ws))
    for _, outs, _, _ in jobs:
        for t in outs.values():
            t.zero_()
    torch.cuda.synchronize()
    for _ in range(10):
        for (run, _, _, _), side in zip(jobs, sides):
            run(side)
    torch.cuda.synchronize()
    for _, outs, want, ws in jobs:
        assert all(kdn.kdn_get_device_status(w) == 0 for w in ws)
        for n, t in outs.items():
            assert torch.equal(t, want[n]), n
