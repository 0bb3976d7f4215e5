"""``stream=`` other than the current one: results that a call makes are recorded on that stream, and
the workspace it makes comes from that stream's own pool, so that their memory is not handed on
while the stream still works there."""
import contextlib
import types

import pytest
import torch

import paper_2609_07816_gb300 as kdn
from test_binding_cpu import BF, FNS, acts, fake, fake_tensor, state  # noqa: F401


@pytest.mark.parametrize("variant", ["diag", "iso"])
def test_everything_made_is_recorded(fake, monkeypatch, variant):  # noqa: F811
    seen = []
    monkeypatch.setattr(torch.Tensor, "record_stream", lambda t, s: seen.append((t, s)), raising=False)
    monkeypatch.setattr(torch.cuda, "ExternalStream", lambda handle: ("external", handle))
    pool, scratch = [None], []

    @contextlib.contextmanager
    def under(stream):
        pool[0], before = stream, pool[0]
        yield
        pool[0] = before

    monkeypatch.setattr(torch.cuda, "stream", under)
    alloc = kdn.alloc_workspace
    monkeypatch.setattr(kdn, "alloc_workspace", lambda *a, **kw: scratch.append(pool[0]) or alloc(*a, **kw))
    st = types.SimpleNamespace(cuda_stream=7)
    fwd, bwd, fsave, bsaved, beff, dec = FNS[variant]
    B, T, H, d = 2, 150, 3, 128
    x = acts(variant, B, T, H, d, d)
    S, p = state(variant, B, H, d, d)
    dO = torch.empty(B, T, H, d, dtype=BF, device="cuda")
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")

    def made(n, w, fn, *a, **kw):  # n results and w workspaces of the call's own
        seen.clear()
        scratch.clear()
        out = fn(*a, **kw)
        assert not seen and scratch == [None] * w  # the current stream: nothing to record
        scratch.clear()
        fn(*a, stream=st, **kw)
        assert len(seen) == n and all(s == ("external", 7) for _, s in seen), fn
        assert scratch == [("external", 7)] * w, fn
        return out

    made(3, 1, fwd, *x)
    made(1, 1, fwd, *x, want_state=False)
    made(1, 0, fwd, *x, want_state=False, workspace=ws)
    saved = made(4, 1, fsave, *x)[3]
    made(6, 1, bsaved, *x, saved, dO, want_state_grads=False)
    made(9, 0, bsaved, *x, saved, dO, workspace=ws)
    grads = made(9, 1, bwd, *x, S, p, dO)
    made(0, 1, bwd, *x, S, p, dO, grads=grads)
    made(1, 0, beff, x[1], x[2], x[3], x[5], saved)
    made(1, 0, dec, *[t[:, 0].contiguous() for t in x], S, p)


@pytest.mark.gpu
@pytest.mark.parametrize("T", [2047, 449])
def test_memory_is_not_handed_on_early(T):
    from paper_2609_07816_gb300 import build
    build.build()
    from kdn_gpu_util import to_dev
    from test_gpu_split import GRADS, NAMES, _case
    ins, _, _ = _case(1, T, 14, 3, "post", False)
    d = to_dev(ins)
    x = [d[n] for n in NAMES]
    kw = dict(out_dtype=BF)
    o, ST, pT, saved = kdn.kdn_diag_fwd_save(*x, **kw)
    gr = kdn.kdn_diag_bwd_saved(*x, saved, d["dO"], want_state_grads=False, **kw)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()

    def over():  # what the allocator hands on next is written over at once
        for n in (1 << 20, 1 << 23, 1 << 26):
            for _ in range(4):
                torch.full((n,), 255, dtype=torch.uint8, device="cuda")

    for _ in range(3):
        # (the side stream waits for the current one before each call: the results' memory comes from there)
        with torch.cuda.stream(side):
            torch.cuda._sleep(20_000_000)
        side.wait_stream(torch.cuda.current_stream())
        got = [kdn.kdn_diag_fwd(*x, stream=side, **kw)]
        over()
        side.wait_stream(torch.cuda.current_stream())
        got.append(kdn.kdn_diag_fwd_save(*x, stream=side, **kw))
        over()
        side.wait_stream(torch.cuda.current_stream())
        g2 = kdn.kdn_diag_bwd_saved(*x, got[1][3], d["dO"], want_state_grads=False, stream=side, **kw)
        over()
        torch.cuda.synchronize()
        for a in got:
            for u, v in zip(a, (o, ST, pT)):
                assert torch.equal(u, v)
        for n in GRADS:
            assert torch.equal(g2[n], gr[n]), n
