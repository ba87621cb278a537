"""The work that a program using this library has it do, as measurable cases.

A case is one pass through the public entry points: a decode step, a forward
(prefill), a training pass (forward that keeps its intermediates, then the
backward that reads them), or the q, k activation and normalisation with its
backward.  Inputs follow the library's own recipe: unit q and k rows, normal v
and upstream gradients, log-decays from the Mamba-2 style gate, sigmoid rates,
states N(0, 0.02^2).
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2509_25223_gb300 as rdn

CLIP = 1.0
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
DEV = "cuda"


def listed():
    return [
        # one user's next token: the smallest call, launch and host latency count
        dict(name="decode_one", op="decode", variant="rdn", N=1, H=16, D=128, dtype="bf16"),
        # a serving batch's next tokens (the benchmark's decode step): states stream from HBM
        dict(name="decode_batch", op="decode", variant="rdn", N=256, H=16, D=128, dtype="bf16"),
        # the smallest sequence call: two fp32 heads of 64, an evaluation or a unit of a small model
        dict(name="forward_f32_small", op="forward", variant="rla", B=1, T=256, H=2, D=64,
             dtype="f32", states=False, seqs=0),
        # one chat prompt of an odd length, continued from states and handing states on
        dict(name="prompt_ragged", op="forward", variant="rdn", B=1, T=777, H=16, D=128,
             dtype="bf16", states=True, seqs=0),
        # prefill of a batch of prompts (the benchmark's forward)
        dict(name="prefill_batch", op="forward", variant="rdn", B=8, T=2048, H=16, D=128,
             dtype="bf16", states=False, seqs=0),
        # long documents, few sequences (the benchmark's long-context forward)
        dict(name="prefill_long", op="forward", variant="rdn", B=2, T=16384, H=16, D=128,
             dtype="bf16", states=True, seqs=0),
        # the benchmark's training pass
        dict(name="train_batch", op="train", variant="rdn", B=8, T=4096, H=16, D=128,
             dtype="bf16", states=False, seqs=0, qk_norm=False),
        # pretraining on packed documents: 15 sequences of 200 to 10,000 tokens in one row
        dict(name="train_packed", op="train", variant="rdn", B=1, T=32768, H=16, D=128,
             dtype="bf16", states=False, seqs=15, qk_norm=False),
        # the additive variant on a small batch of ragged length, raw q and k normalised in the call
        dict(name="train_rla_norm", op="train", variant="rla", B=2, T=2000, H=16, D=128,
             dtype="bf16", states=True, seqs=0, qk_norm=True),
        # training with heads of 64, the other head size in common use
        dict(name="train_d64", op="train", variant="rdn", B=4, T=2048, H=16, D=64,
             dtype="bf16", states=False, seqs=0, qk_norm=False),
        # training in full fp32, ragged length
        dict(name="train_f32", op="train", variant="rdn", B=2, T=1000, H=8, D=128,
             dtype="f32", states=True, seqs=0, qk_norm=False),
        # the standalone activation and normalisation of q and k, both directions
        dict(name="prologue", op="prologue", B=8, T=4096, H=16, D=128, dtype="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["decode", "forward", "forward", "train", "train", "train", "prologue"])
    H = rng.choice([2, 4, 5, 8, 12, 16])
    if op == "decode":
        return dict(op=op, variant=rng.choice(["rdn", "rla"]), N=_log_int(rng, 1, 256), H=H,
                    D=rng.choice([64, 128]), dtype=rng.choice(["bf16", "bf16", "f32"]))
    if op == "prologue":
        return dict(op=op, B=rng.randint(1, 8), T=_log_int(rng, 64, 4096), H=H,
                    D=rng.choice([64, 128]), dtype=rng.choice(["bf16", "f32"]))
    kind = rng.choice(["bf16_128", "bf16_128", "bf16_64", "f32_64", "f32_128"])
    dtype, D = kind.split("_")
    # tokens x heads at most those of the largest listed case of the kind
    most = {"bf16_128": 8 * 4096 * 16, "bf16_64": 4 * 2048 * 16, "f32_64": 4 * 2048 * 16,
            "f32_128": 2 * 1000 * 8}[kind]
    T = _log_int(rng, 64, min(16384 if op == "forward" else 4096, most // H))
    B = max(1, min(8, _log_int(rng, 1, 8), most // (T * H)))
    seqs = rng.randint(2, 12) if B == 1 and T > 256 and rng.random() < 0.5 else 0
    case = dict(op=op, variant=rng.choice(["rdn", "rdn", "rla"]), B=B, T=T, H=H, D=int(D),
                dtype=dtype, states=rng.random() < 0.5, seqs=seqs)
    if op == "train":
        case["qk_norm"] = rng.random() < 0.3
    return case


def _lengths(case):
    """The token counts of the case's sequences: B equal ones, or `seqs` packed
    documents of log-uniform lengths that fill the row."""
    if not case["seqs"]:
        return [case["T"]] * case["B"]
    r = np.random.default_rng(1000 * case["seqs"] + case["T"])
    w = np.exp(r.uniform(0.0, math.log(64.0), case["seqs"]))
    cuts = np.floor(np.cumsum(w) / w.sum() * case["T"]).astype(int)
    cuts[-1] = case["T"]
    return [int(n) for n in np.diff(np.concatenate([[0], cuts]))]


def _normalise(x, eps=1e-12):
    u = F.silu(x)
    return u / u.norm(dim=-1, keepdim=True).clamp_min(eps)


def _gates(randn, variant, *shape):
    x = randn(*shape)
    return dict(g=F.logsigmoid(x) if variant == "rla" else -F.softplus(x),
                beta=torch.sigmoid(randn(*shape)), gamma=torch.sigmoid(randn(*shape)))


def _off_the_clip(case, x, lens, margin=2e-3):
    """Moves the few elements of v whose residual lies within `margin` of the
    clip threshold past it.  The gradient jumps there, so that two right answers
    would differ by whether rounding put an element on one side or the other."""
    N, L = len(lens), max(lens)
    H, D = case["H"], case["D"]
    first = np.concatenate([[0], np.cumsum(lens)[:-1]])
    at = torch.from_numpy(first).to(DEV)
    last = torch.from_numpy(first + np.array(lens) - 1).to(DEV)
    flat = lambda t: t.reshape(case["B"] * case["T"], *t.shape[2:])  # noqa: E731
    k = flat(x["k"]).float()
    if case.get("qk_norm"):
        k = _normalise(k).to(x["k"].dtype).float()
    v, beta, alpha = flat(x["v"]).clone(), flat(x["beta"]), flat(x["g"]).exp()
    S = torch.zeros(N * H, D, D, device=DEV) if x["S0"] is None else x["S0"].reshape(N * H, D, D).clone()
    for t in range(L):
        row = torch.minimum(at + t, last)  # a sequence that has ended repeats its last token, unchanged
        kt = k[row].reshape(N * H, 1, D)
        vt = v[row].reshape(N * H, 1, D).float()
        p = torch.bmm(kt, S)
        r = vt - p
        near = ((r.abs() - CLIP).abs() < margin) & (at + t <= last).repeat_interleave(H)[:, None, None]
        moved = p + torch.sign(r) * (CLIP + 2 * margin + vt.abs() / 256)
        vt = torch.where(near, moved, vt).to(v.dtype)
        v[row] = vt.reshape(N, H, D)
        vt = vt.float()
        a = alpha[row].reshape(N * H, 1, 1)
        b = beta[row].reshape(N * H, 1, 1)
        e = vt - a * p if case["variant"] == "rdn" else vt
        S = torch.baddbmm(a * S, (b * kt).transpose(1, 2), e)
    return v.reshape(x["v"].shape)


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)

    def randn(*shape):
        return torch.randn(*shape, generator=gen, device=DEV)

    H, D, dt = case["H"], case["D"], DTYPES[case["dtype"]]
    st = {"case": case}
    if case["op"] == "decode":
        N = case["N"]
        st["S"], st["R"] = 0.02 * randn(N, H, D, D), 0.02 * randn(N, H, D, D)
        for n in ("q", "k"):
            st[n] = F.normalize(randn(N, H, D), dim=-1).to(dt)
        st["v"] = randn(N, H, D).to(dt)
        st.update(_gates(randn, case["variant"], N, H))
        return st
    B, T = case["B"], case["T"]
    if case["op"] == "prologue":
        for n in ("q", "k", "dq", "dk"):
            st[n] = randn(B, T, H, D).to(dt)
        return st
    raw = case.get("qk_norm", False)
    for n in ("q", "k"):
        x = randn(B, T, H, D)
        st[n] = (x if raw else F.normalize(x, dim=-1)).to(dt)
    st["v"] = randn(B, T, H, D).to(dt)
    st.update(_gates(randn, case["variant"], B, T, H))
    lens = _lengths(case)
    st["S0"] = st["R0"] = st["cu"] = None
    if case["states"]:
        st["S0"], st["R0"] = 0.02 * randn(len(lens), H, D, D), 0.02 * randn(len(lens), H, D, D)
    if case["seqs"]:
        st["cu"] = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32, device=DEV)
    train = case["op"] == "train"

    def space(what, **kw):
        n = rdn.workspace_bytes(case["variant"] + what, B, T, H, D, dtype=dt, cu_seqlens=st["cu"],
                                qk_norm=raw, **kw)
        return torch.empty(n, dtype=torch.uint8, device=DEV)

    st["ws_fwd"] = space("_fwd", save_for_bwd=train)  # kept between calls, as a program would
    if train:
        st["dO"] = randn(B, T, H, D).to(dt)
        st["v"] = _off_the_clip(case, st, lens)
        st["ws_bwd"] = space("_bwd")
    return st


def run(st):
    case = st["case"]
    if case["op"] == "decode":
        o = rdn.rdn_decode_step(st["q"], st["k"], st["v"], st["g"], st["beta"], st["gamma"],
                                st["S"], st["R"], clip=CLIP, variant=case["variant"])
        return {"o": o, "S": st["S"], "R": st["R"]}
    if case["op"] == "prologue":
        yq, yk = rdn.qk_prologue(st["q"], st["k"])
        dq, dk = rdn.qk_prologue_bwd(st["q"], st["k"], st["dq"], st["dk"])
        return {"yq": yq, "yk": yk, "dq": dq, "dk": dk}
    x = [st[n] for n in ("q", "k", "v", "g", "beta", "gamma")]
    fwd, bwd = (rdn.rdn_fwd, rdn.rdn_bwd) if case["variant"] == "rdn" else (rdn.rla_fwd, rdn.rla_bwd)
    opt = dict(clip=CLIP, S0=st["S0"], R0=st["R0"], cu_seqlens=st["cu"])
    if case["op"] == "forward":
        o, ST, RT = fwd(*x, workspace=st["ws_fwd"], **opt)
        return {"o": o, "ST": ST, "RT": RT}
    opt["qk_norm"] = case["qk_norm"]
    o, ST, RT, Sc, Rc = fwd(*x, workspace=st["ws_fwd"], return_chunk_states=True,
                            save_for_bwd=True, **opt)
    grads = bwd(*x, st["dO"], S_chunks=Sc, R_chunks=Rc, workspace=st["ws_bwd"],
                fwd_workspace=st["ws_fwd"], fwd_saved=True, **opt)
    return {"o": o, "ST": ST, "RT": RT, **grads}


def work(case):
    """Each input read once and each output written once; the recurrence's own
    products, 2 D^2 flops each: S and R read with k and q and updated (6 per
    token and head; 5 for RLA, whose R is not read with k), twice that again
    for the backward."""
    D, esz = case["D"], 2 if case["dtype"] == "bf16" else 4
    per = 12 * D * D if case.get("variant") != "rla" else 10 * D * D
    if case["op"] == "decode":
        nh = case["N"] * case["H"]
        return {"bytes": nh * (16 * D * D + 4 * D * esz + 12), "flops": nh * per}
    rows = case["B"] * case["T"] * case["H"]
    if case["op"] == "prologue":  # x in, y out; x, dy in, dx out; for q and k
        return {"bytes": 2 * rows * D * esz * 5, "flops": 2 * rows * D * 20}
    states = len(_lengths(case)) * case["H"] * D * D * 4 * 2
    if case["op"] == "forward":
        return {"bytes": rows * (4 * D * esz + 12) + states * (2 if case["states"] else 1),
                "flops": rows * per}
    # q, k, v, dO, o, dq, dk, dv; the gates and their gradients; states out, their gradients out
    return {"bytes": rows * (8 * D * esz + 24) + states * (3 if case["states"] else 2),
            "flops": 3 * rows * per}


class _Held(torch.autograd.Function):
    """Normalised rows as they are held, in the inputs' type; the gradient passes."""

    @staticmethod
    def forward(ctx, y, dtype):
        return y.to(dtype).double()

    @staticmethod
    def backward(ctx, dy):
        return dy, None


def _sequences(variant, q, k, v, g, beta, gamma, S, R):
    """The layer over [N, H, L, D] sequences in 64 bits, 64 tokens at a time."""
    N, H, L, D = q.shape
    out = []
    for t0 in range(0, L, 64):
        qc, kc, vc = (x[:, :, t0:t0 + 64] for x in (q, k, v))
        gc, bc, mc = (x[:, :, t0:t0 + 64] for x in (g, beta, gamma))
        n = qc.shape[2]
        b = gc.cumsum(-1)
        Gam, Gprev = b.exp()[..., None], (b - gc).exp()[..., None]
        upper = torch.ones(n, n, dtype=torch.bool, device=q.device).triu(1)
        dec = (b[..., :, None] - b[..., None, :]).masked_fill(upper, -math.inf).exp()
        decp = ((b - gc)[..., :, None] - b[..., None, :]).masked_fill(~upper.T, -math.inf).exp()
        KK, QK = kc @ kc.transpose(-1, -2), qc @ kc.transpose(-1, -2)
        end = (b[..., -1:] - b).exp()

        def solve(rate, x, state):
            if variant == "rla":
                return x
            A = dec * rate[..., None, :] * KK
            return torch.linalg.solve_triangular(A, x - Gam * (kc @ state), upper=False,
                                                 unitriangular=True)

        E = solve(bc, vc, S)
        P = Gprev * (kc @ S) + (decp * bc[..., None, :] * KK) @ E
        base = Gam * (qc @ S) + ((dec * bc[..., None, :] * QK).tril(-1)) @ E
        r = (vc - P).clamp(-CLIP, CLIP)
        E2 = solve(mc, r, R)
        aux = Gam * (qc @ R) + (dec * mc[..., None, :] * QK) @ E2
        out.append(base + mc[..., None] * aux)
        carry = Gam[:, :, -1:]
        S = carry * S + kc.transpose(-1, -2) @ ((bc * end)[..., None] * E)
        R = carry * R + kc.transpose(-1, -2) @ ((mc * end)[..., None] * E2)
    return torch.cat(out, 2), S, R


def exact(case, seed):
    st = prepare(case, seed)
    st.pop("ws_fwd", None), st.pop("ws_bwd", None)
    d = lambda t: None if t is None else t.double()  # noqa: E731
    if case["op"] == "decode":
        q, k, v, S, R = (d(st[n]) for n in ("q", "k", "v", "S", "R"))
        a, b, m = (x.double()[..., None, None] for x in (st["g"].double().exp(), st["beta"], st["gamma"]))
        q, k, v = q[..., None, :], k[..., None, :], v[..., None, :]
        p, kR = k @ S, k @ R
        r = (v - p).clamp(-CLIP, CLIP)
        e, e2 = (v - a * p, r - a * kR) if case["variant"] == "rdn" else (v, r)
        o = a * (q @ S)
        S = a * S + b * k.transpose(-1, -2) @ e
        R = a * R + m * k.transpose(-1, -2) @ e2
        return {"o": (o + m * (q @ R))[..., 0, :], "S": S, "R": R}
    if case["op"] == "prologue":
        got = {}
        for n in ("q", "k"):
            x = d(st[n]).requires_grad_()
            y = _normalise(x)
            y.backward(d(st["d" + n]))
            got["y" + n], got["d" + n] = y.detach(), x.grad
        return got
    train = case["op"] == "train"
    H, D, lens = case["H"], case["D"], _lengths(case)
    names = ("q", "k", "v", "g", "beta", "gamma")
    same = len(set(lens)) == 1
    groups = [(0, len(lens), lens[0])] if same else [(i, 1, n) for i, n in enumerate(lens)]
    parts, tok = [], 0
    for s0, n, L in groups:
        def seq(t):  # [n, H, L, ...] of this group's tokens
            t = t.reshape(-1, *t.shape[2:])[tok:tok + n * L].double()
            return t.reshape(n, L, *t.shape[1:]).transpose(1, 2)

        x = {m: seq(st[m]).detach().requires_grad_(train) for m in names}
        S0, R0 = ((torch.zeros(n, H, D, D, dtype=torch.float64, device=DEV) if st[m] is None
                   else st[m][s0:s0 + n].double()).requires_grad_(train) for m in ("S0", "R0"))
        y = dict(x)
        if case.get("qk_norm"):
            for m in ("q", "k"):
                y[m] = _Held.apply(_normalise(x[m]), st[m].dtype)
        o, ST, RT = _sequences(case["variant"], *(y[m] for m in names), S0, R0)
        back = lambda t: t.detach().transpose(1, 2).reshape(n * L, *t.shape[1:2], *t.shape[3:])  # noqa: E731
        got = {"o": back(o), "ST": ST.detach(), "RT": RT.detach()}
        if train:
            o.backward(seq(st["dO"]))
            got.update({"d" + m: back(x[m].grad) for m in names})
            got["dS0"] = S0.grad
            got["dR0"] = R0.grad
        parts.append(got)
        tok += n * L
    got = {m: torch.cat([p[m] for p in parts]) for m in parts[0]}
    for m in got:
        if m not in ("ST", "RT", "dS0", "dR0"):
            got[m] = got[m].reshape(case["B"], case["T"], *got[m].shape[1:])
    return got
