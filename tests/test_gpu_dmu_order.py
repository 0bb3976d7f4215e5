"""dmu of the general backward: the chunks' parts are added in one order, so that it repeats
exactly, and as many as eight blocks of chunks are all in it."""
import numpy as np
import pytest
import torch

import oracle
from kdn_gpu_util import check, to_dev
from kdn_inputs import make_inputs

pytestmark = pytest.mark.gpu
NAMES = ("q", "k", "v", "g", "omega", "r")


@pytest.mark.parametrize("variant,T", [("diag", 1), ("diag", 1500), ("iso", 33), ("iso", 1500)])
def test_dmu_repeats(variant, T):
    from paper_2609_07816_gb300 import build
    build.build()
    import paper_2609_07816_gb300 as kdn
    ins = make_inputs(variant, 2, T, 5, 64, 32, dtype="f32", seed=T, s0_std=0.1, p0_range=(0.5, 2.0),
                      per_channel_decay=variant == "diag", with_grad=True)
    d = to_dev(ins)
    bwd = kdn.kdn_diag_bwd if variant == "diag" else kdn.kdn_iso_bwd
    run = lambda: bwd(*[d[n] for n in NAMES], d["S0"], d["p0"], d["dO"])["dmu"]
    first = run()
    for _ in range(20):
        assert torch.equal(run(), first)
    ref = oracle.bwd(variant, *[ins[n] for n in NAMES], ins["S0"], ins["p0"], ins["dO"])
    check("dmu", first, ref["dmu"], "f32")
    assert np.isfinite(ref["dmu"]).all()
