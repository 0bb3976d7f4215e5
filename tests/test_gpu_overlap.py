"""Gradient buffers that take the place of their inputs, or that serve twice: the diagonal
backward uses the gradient buffers as scratch only where nothing it reads lies there."""
import pytest
import torch

from kdn_gpu_util import to_dev
from test_gpu_split import GRADS, NAMES, _case

pytestmark = pytest.mark.gpu
INPUT = dict(zip(GRADS, NAMES))


@pytest.mark.parametrize("T", [512, 449])
@pytest.mark.parametrize("gates", ["post", "logits"])
@pytest.mark.parametrize("over", [{"dv": "dO"}, {"dq": "q"}, {"dk": "k"}, {"domega": "omega"}, {"dr": "r"},
                                  {"dq": "q", "dk": "k", "dv": "v", "dg": "g", "domega": "omega", "dr": "r"},
                                  {"dg": "dq"}], ids=lambda o: "-".join(o))
def test_gradients_over_inputs(over, gates, T):
    from paper_2609_07816_gb300 import build
    build.build()
    import paper_2609_07816_gb300 as kdn
    ins, _, _ = _case(2, T, 6, T, gates, False)
    G = kdn.KDN_GATES_LOGITS if gates == "logits" else kdn.KDN_GATES_POST
    kw = dict(out_dtype=torch.bfloat16, gates=G)

    def run(over):
        d = to_dev(ins)
        x = [d[n] for n in NAMES]
        _, _, _, saved = kdn.kdn_diag_fwd_save(*x, d["S0"], d["p0"], **kw)
        grads = {n: torch.empty_like(d[INPUT[n]]) for n in GRADS}
        for n, at in over.items():
            grads[n] = grads[at] if at in grads else d[at]
        gr = kdn.kdn_diag_bwd_saved(*x, saved, d["dO"], grads=grads, want_state_grads=False, **kw)
        return {n: t for n, t in gr.items() if n not in over or over[n] not in grads}

    apart, got = run({}), run(over)
    torch.cuda.synchronize()
    for n, t in got.items():
        if not any(at == n for at in over.values()):  # (a buffer that serves twice holds either gradient)
            assert torch.equal(t, apart[n]), n
