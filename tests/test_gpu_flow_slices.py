"""The parallel forward of few sequences beyond one slice of its workspace: the state goes from
launch to launch in float32, so the results are those of the one-kernel forward bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# slices of 64, 56 and 409 chunks at most; fast: some channels leave the referenced decay range
@pytest.mark.parametrize("B,T,H,gates,fast", [(2, 5000, 16, "logits", False), (2, 8256, 16, "post", True),
                                              (4, 3649, 9, "post", False), (1, 28801, 5, "post", True)])
@pytest.mark.parametrize("state", [False, True])
def test_slices_equal_the_one_kernel(B, T, H, gates, fast, state):
    from paper_2609_07816_gb300 import build
    build.build()
    import paper_2609_07816_gb300 as kdn
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T)
    F = torch.nn.functional
    n = lambda *s: torch.randn(*s, device="cuda", generator=gen)
    g, w, r = n(B, T, H, 128) + 3, n(B, T, H, 128), n(B, T, H)
    if gates == "post":
        g, w, r = F.logsigmoid(g), F.softplus(w), F.softplus(r) + 0.05
        if fast:
            g[:, T // 3:, :, ::5] = -9.0
    x = [t.bfloat16() for t in (F.normalize(n(B, T, H, 128), dim=-1), F.normalize(n(B, T, H, 128), dim=-1),
                                n(B, T, H, 128), g, w, r)]
    st = (n(B, H, 128, 128) * 0.05, torch.rand(B, H, 128, device="cuda", generator=gen) + 0.5) if state else (None, None)
    G = kdn.KDN_GATES_LOGITS if gates == "logits" else kdn.KDN_GATES_POST
    kw = dict(out_dtype=torch.bfloat16, gates=G)
    desc = kdn.make_desc(B, T, H, 128, 128, torch.bfloat16, **kw)
    ws = kdn.alloc_workspace(desc, 0)
    assert 66560 * B * H < ws.numel() < 66560 * B * H * (T // 64)  # slices
    many = kdn.kdn_diag_fwd(*x, *st, workspace=ws, **kw)
    one = kdn.kdn_diag_fwd(*x, *st, workspace=torch.empty(256, dtype=torch.uint8, device="cuda"), **kw)
    bare, _, _ = kdn.kdn_diag_fwd(*x, *st, workspace=ws, want_state=False, **kw)
    torch.cuda.synchronize()
    assert kdn.kdn_get_device_status(ws) == 0
    for u, v in zip(many, one):
        assert torch.equal(u, v)
    assert torch.equal(bare, one[0])
