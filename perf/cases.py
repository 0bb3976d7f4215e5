"""The calls whose speed counts, as a user of this package makes them.

A Kalman Delta Network layer is called in three ways: one decode step for a batch
of running sequences, a forward over a prompt (prefill), and a training step
(forward and backward).  The cases cover both variants (Diagonal and Isotropic),
bfloat16 and float32 activations, both gate forms, ragged lengths and the sizes
of the repository's benchmark and parity tests.  Inputs follow the recipe of
``kdn_inputs.py`` (normalised q and k, decay sigmoid(N(m, 1)), softplus noises),
drawn on the device.

A case's fields:
  op       "decode", "prefill" or "train"
  variant  "diag" or "iso" (iso: one decay per head, or per channel)
  B, T, H, dk, dv   sizes (decode has no T)
  dtype, out_dtype  stored types of the activations and of o / the gradients
  gates    "post" (log alpha, omega, r) or "logits"
  decay    mean m of the decay logit: 2 forgets within tens of tokens, 6 keeps
           the memory over thousands
  state    prefill: starts from a memory and an uncertainty; train: also returns
           the gradients of the initial state and of mu
"""
import math

import torch

import paper_2609_07816_gb300 as kdn

_DT = {"bf16": torch.bfloat16, "f32": torch.float32}
_GATES = {"post": kdn.KDN_GATES_POST, "logits": kdn.KDN_GATES_LOGITS}
_NAMES = ("q", "k", "v", "g", "omega", "r")
_GRADS = ("dq", "dk", "dv", "dg", "domega", "dr")


def _case(name, op, variant, B, T, H, d, *, dv=None, dtype="bf16", out_dtype="bf16",
          gates="post", decay=2, state=False, per_channel=None):
    c = dict(op=op, variant=variant, B=B, T=T, H=H, dk=d, dv=d if dv is None else dv, dtype=dtype,
             out_dtype=out_dtype, gates=gates, decay=decay, state=state,
             per_channel=variant == "diag" if per_channel is None else per_channel)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one user generating text: the smallest call there is, once per layer and token
        _case("decode_diag_one", "decode", "diag", 1, 1, 16, 128),
        # a serving batch of 256 running sequences, bound by the memories themselves
        _case("decode_diag_batch", "decode", "diag", 256, 1, 16, 128, out_dtype="f32"),
        # a smaller serving batch of the isotropic layer with the gate logits as they come
        _case("decode_iso_batch", "decode", "iso", 64, 1, 12, 128, gates="logits"),
        # one user's prompt of odd length ahead of decoding
        _case("prefill_diag_prompt", "prefill", "diag", 1, 777, 16, 128, gates="logits"),
        # a batch of full-length prompts, or scoring
        _case("prefill_diag_batch", "prefill", "diag", 8, 4096, 16, 128),
        # one very long document, continued from a memory
        _case("prefill_diag_long", "prefill", "diag", 1, 65536, 16, 128, state=True),
        # a long document through the isotropic layer with a slow decay
        _case("prefill_iso_long", "prefill", "iso", 1, 32768, 12, 128, decay=6),
        # a head width that the bf16 tensor-core kernels do not serve
        _case("prefill_diag_d64", "prefill", "diag", 8, 2048, 16, 64),
        # the training step of the 1.3B-parameter model's layer
        _case("train_diag", "train", "diag", 8, 4096, 16, 128),
        # the training step of the 750M-parameter model's layer
        _case("train_iso", "train", "iso", 8, 2048, 12, 128),
        # training on a small batch of odd length, logit gates, a slow decay
        _case("train_diag_ragged", "train", "diag", 2, 1999, 16, 128, gates="logits", decay=6),
        # training a small model in float32
        _case("train_diag_f32", "train", "diag", 2, 1024, 8, 64, dtype="f32", out_dtype="f32",
              state=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("decode", "prefill", "prefill", "train", "train"))
    variant = rng.choice(("diag", "diag", "iso"))
    H = rng.choice((4, 8, 12, 16, 16, 24, 32))
    d = rng.choice((32, 64, 128, 128, 128, 128))
    dv = rng.choice((d, d, d, rng.choice((32, 64, 128))))
    dtype = rng.choice(("bf16", "bf16", "bf16", "f32"))
    out_dtype = "f32" if dtype == "f32" else rng.choice(("bf16", "bf16", "f32"))
    gates = rng.choice(("post", "logits"))
    decay = rng.choice((2, 2, 4, 6))
    per_channel = variant == "diag" or rng.random() < 0.25
    state = rng.random() < 0.3
    fused = dtype == "bf16" and d == 128 and dv == 128
    if op == "decode":
        B, T = _log_int(rng, 1, 4096 // H), 1
    else:
        # token-heads of one call; the general kernels are called with smaller problems
        cap = (1 << 19 if op == "train" else 1 << 20) if fused else 1 << 17
        T = _log_int(rng, 16, min(cap // H, 65536 if op == "prefill" else 16384))
        B = _log_int(rng, 1, max(1, min(64, cap // (H * T))))
        if rng.random() < 0.3 and T > 64:
            T -= T % 64
    return _case(None, op, variant, B, T, H, d, dv=dv, dtype=dtype, out_dtype=out_dtype,
                 gates=gates, decay=decay, state=state, per_channel=per_channel)


def _inputs(case, seed):
    """The tensors a layer has in hand when it calls the mixer."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(*shape, device="cuda", generator=gen)

    def uniform(lo, hi, *shape):
        return torch.rand(*shape, device="cuda", generator=gen) * (hi - lo) + lo

    B, T, H, dk, dv = (case[n] for n in ("B", "T", "H", "dk", "dv"))
    diag, post, dt = case["variant"] == "diag", case["gates"] == "post", _DT[case["dtype"]]
    tok = (B, H) if case["op"] == "decode" else (B, T, H)
    F = torch.nn.functional
    x = {"q": F.normalize(normal(*tok, dk), dim=-1), "k": F.normalize(normal(*tok, dk), dim=-1),
         "v": normal(*tok, dv)}
    g = normal(*tok, *((dk,) if case["per_channel"] else ())) + case["decay"]
    w = normal(*tok, *((dk,) if diag else ()))
    r = normal(*tok)
    x["g"], x["omega"], x["r"] = (F.logsigmoid(g), F.softplus(w), F.softplus(r)) if post else (g, w, r)
    x = {n: t.to(dt) for n, t in x.items()}
    pshape = (B, H, dk) if diag else (B, H)
    if case["op"] == "decode" or case["state"]:
        x["S0"] = normal(B, H, dk, dv) * 0.02
        x["p0"] = uniform(0.5, 2.0, *pshape)
    else:
        x["S0"] = x["p0"] = None
    if case["op"] == "train":
        x["dO"] = normal(*tok, dv).to(dt)
    return x


def _saves_context(case):
    """The training pair that keeps a context serves bf16 at dk = dv = 128."""
    return case["dtype"] == "bf16" and case["dk"] == 128 and case["dv"] == 128


def prepare(case, seed):
    x = _inputs(case, seed)
    st = dict(case=case, x=[x[n] for n in _NAMES], S0=x["S0"], p0=x["p0"], dO=x.get("dO"),
              kw=dict(out_dtype=_DT[case["out_dtype"]], gates=_GATES[case["gates"]]))
    if case["op"] == "decode":
        return st
    variant = 0 if case["variant"] == "diag" else 1
    desc = kdn.make_desc(case["B"], case["T"], case["H"], case["dk"], case["dv"], _DT[case["dtype"]],
                         decay_per_channel=int(case["per_channel"]), out_dtype=st["kw"]["out_dtype"],
                         gates=st["kw"]["gates"])
    # scratch and, for training, the saved context: a program keeps them from step to step
    st["ws"] = kdn.alloc_workspace(desc, variant, False)
    if case["op"] == "train":
        if _saves_context(case):
            st["saved"] = torch.empty(kdn.saved_bytes(desc, variant), dtype=torch.uint8, device="cuda")
        else:
            st["ws_b"] = kdn.alloc_workspace(desc, variant, True)
    return st


def run(state):
    c, x, kw = state["case"], state["x"], state["kw"]
    diag = c["variant"] == "diag"
    if c["op"] == "decode":
        step = kdn.kdn_diag_decode_step if diag else kdn.kdn_iso_decode_step
        o = step(*x, state["S0"], state["p0"], **kw)
        return {"o": o, "S": state["S0"], "p": state["p0"]}
    if c["op"] == "prefill":
        fwd = kdn.kdn_diag_fwd if diag else kdn.kdn_iso_fwd
        o, ST, pT = fwd(*x, state["S0"], state["p0"], workspace=state["ws"], **kw)
        return {"o": o, "S": ST, "p": pT}
    if "saved" in state:
        save = kdn.kdn_diag_fwd_save if diag else kdn.kdn_iso_fwd_save
        bwd = kdn.kdn_diag_bwd_saved if diag else kdn.kdn_iso_bwd_saved
        o, _, _, saved = save(*x, state["S0"], state["p0"], saved=state["saved"], want_state=False,
                              workspace=state["ws"], **kw)
        grads = bwd(*x, saved, state["dO"], want_state_grads=c["state"], workspace=state["ws"], **kw)
    else:
        fwd = kdn.kdn_diag_fwd if diag else kdn.kdn_iso_fwd
        bwd = kdn.kdn_diag_bwd if diag else kdn.kdn_iso_bwd
        o, _, _ = fwd(*x, state["S0"], state["p0"], want_state=False, workspace=state["ws"], **kw)
        grads = bwd(*x, state["S0"], state["p0"], state["dO"], want_state_grads=c["state"],
                    workspace=state["ws_b"], **kw)
    return {"o": o, **grads}


def work(case):
    B, T, H, dk, dv = (case[n] for n in ("B", "T", "H", "dk", "dv"))
    diag, th = case["variant"] == "diag", B * T * H
    es = 2 if case["dtype"] == "bf16" else 4
    os_ = 2 if case["out_dtype"] == "bf16" else 4
    gates = (dk if case["per_channel"] else 1) + (dk if diag else 1) + 1  # g, omega, r
    elems = 2 * dk + dv + gates                                           # one token-head's inputs
    st = B * H * (dk * dv + (dk if diag else 1)) * 4
    if case["op"] == "decode":
        b = th * (elems * es + dv * os_) + 2 * st
    elif case["op"] == "prefill":
        b = th * (elems * es + dv * os_) + st * (2 if case["state"] else 1)
    else:  # the inputs and dO read, o and the gradients written
        b = th * ((elems + dv) * es + (dv + elems) * os_) + (2 * st + 4 * B * H if case["state"] else 0)
    # S^T k, the rank-one write and S^T q of the token recurrence; its adjoint takes twice that
    return {"bytes": b, "flops": th * 6 * dk * dv * (3 if case["op"] == "train" else 1)}


# --- the token recurrence in float64, on plain torch -------------------------------------------

def _gates64(case, g, w, r):
    if case["gates"] == "post":
        return g, w, r
    F = torch.nn.functional
    return F.logsigmoid(g), F.softplus(w), kdn.R_MIN_DEFAULT + F.softplus(r)


def _tokens64(case, q, k, v, g, w, r, S, p, mu):
    """Tokens [t, N, ...] from the state S [N, dk, dv], p: outputs o [t, N, dv], S, p."""
    diag, dk = case["variant"] == "diag", case["dk"]
    tau = 1.0 / math.sqrt(dk)
    g, w, r = _gates64(case, g, w, r)
    al = g.exp() if case["per_channel"] else g.exp().unsqueeze(-1)
    k2 = k * k
    if diag:
        a, u = al * al, mu.unsqueeze(-1) * k2 / r.unsqueeze(-1)
    else:
        n2 = k2.sum(-1)
        a, u = (al * al).mean(-1), mu * n2 / (dk * r)
    hats = []
    for at, wt, ut in zip(a.unbind(0), w.unbind(0), u.unbind(0)):
        h = torch.addcmul(wt, at, p)
        hats.append(h)
        p = h / (1 + ut * h)
    hat = torch.stack(hats)
    if diag:
        kap = hat * k / (r + (hat * k2).sum(-1)).unsqueeze(-1)
    else:
        kap = (hat / (r + hat * n2)).unsqueeze(-1) * k
    outs = []
    for alt, kt, qt, vt, kapt in zip(al.unsqueeze(-1).unbind(0), k.unsqueeze(-2).unbind(0),
                                     (tau * q).unsqueeze(-2).unbind(0), v.unsqueeze(-2).unbind(0),
                                     kap.unsqueeze(-1).unbind(0)):
        D = alt * S
        S = torch.baddbmm(D, kapt, vt - torch.bmm(kt, D))
        outs.append(torch.bmm(qt, S))
    return torch.stack(outs).squeeze(-2), S, p


def exact(case, seed):
    B, T, H, dk, dv = (case[n] for n in ("B", "T", "H", "dk", "dv"))
    N, diag, SEG = B * H, case["variant"] == "diag", 64
    x = _inputs(case, seed)

    def rows(t):  # [B, T, H, ...] -> [T, B*H, ...]
        t = t.double()
        if case["op"] == "decode":
            return t.reshape(1, N, *t.shape[2:])
        return t.transpose(0, 1).reshape(T, N, *t.shape[3:])

    def back(t):  # [T, B*H, ...] -> [B, T, H, ...]
        t = t.reshape(T, B, H, *t.shape[2:])
        return t[0] if case["op"] == "decode" else t.transpose(0, 1)

    ins = [rows(x[n]) for n in _NAMES]
    mu = torch.full((N,), float(dk), dtype=torch.float64, device="cuda")
    S = torch.zeros(N, dk, dv, dtype=torch.float64, device="cuda")
    p = torch.ones(*((N, dk) if diag else (N,)), dtype=torch.float64, device="cuda")
    if x["S0"] is not None:
        S, p = x["S0"].double().reshape(S.shape), x["p0"].double().reshape(p.shape)
    pshape = (B, H, dk) if diag else (B, H)
    train = case["op"] == "train"
    entry, outs = [], []
    with torch.no_grad():
        for t0 in range(0, T, SEG):
            if train:
                entry.append((S, p))
            o, S, p = _tokens64(case, *(t[t0:t0 + SEG] for t in ins), S, p, mu)
            outs.append(o)
    o = back(torch.cat(outs))
    if not train:
        return {"o": o, "S": S.reshape(B, H, dk, dv), "p": p.reshape(pshape)}
    dO = rows(x["dO"])
    dS, dp, dmu = torch.zeros_like(S), torch.zeros_like(p), torch.zeros_like(mu)
    grads = [torch.empty_like(t) for t in ins]
    for t0 in reversed(range(0, T, SEG)):
        S, p = entry.pop()
        leaves = [t[t0:t0 + SEG].detach().requires_grad_() for t in ins]
        leaves += [t.detach().requires_grad_() for t in (S, p, mu)]
        out = _tokens64(case, *leaves)
        got = torch.autograd.grad(out, leaves, (dO[t0:t0 + SEG], dS, dp))
        for full, part in zip(grads, got):
            full[t0:t0 + SEG] = part
        dS, dp = got[6], got[7]
        dmu += got[8]
    res = {"o": o, **{n: back(t) for n, t in zip(_GRADS, grads)}}
    if case["state"]:
        res.update(dS0=dS.reshape(B, H, dk, dv), dp0=dp.reshape(pshape), dmu=dmu.reshape(B, H))
    return res
