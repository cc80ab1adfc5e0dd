"""The measured cases: what a user of this library has it do, through its public entry
points, over the range of sizes, types and modes it is used at.

Sizes come from the repository's own workloads (parser-scale StackLSTMs with H = 200, a
string-to-tree-decoder-like one with H = 1024, a wide batch of deep stacks, the tiny fp32
one, the arc-hybrid parser step) and from odd, ragged sizes between them. A training call
takes the gradient of every step's output (``dy``, as a layer above gives it) or of the
final top alone (``d_top_h``); an inference call returns every step's output. The calls
run in asynchronous mode, as a training loop uses them, or (``wait``) in the default mode,
where each call reports its status before it returns.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1904_03409_gb300 import binding as bd
from paper_1904_03409_gb300 import runner

# ------------------------------------------------------------------------------- cases
_WALK = (1 / 3, 1 / 3, 1 / 3)


def _lstm(name, dtype, T, B, I, H, call="train", loss="steps", ops="arc", push_only=False, wait=False, probs=_WALK,
          ragged=False):
    case = dict(kind="lstm", dtype=dtype, T=T, B=B, I=I, H=H, call=call, loss=loss, ops=ops, push_only=push_only,
                wait=wait, push=probs[0], pop=probs[1], hold=probs[2], ragged=ragged)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest fp32 training call (a gradient check, a toy grammar): latency alone
        _lstm("tiny_fp32", "fp32", 12, 4, 16, 16, loss="top", ops="walk", wait=True),
        # a small full-precision model with sizes that divide nothing
        _lstm("small_fp32", "fp32", 61, 16, 75, 100, ops="walk", probs=(0.5, 0.3, 0.2), ragged=True),
        # full-precision training of a parser's stack at the usual minibatch
        _lstm("parser64_fp32", "fp32", 185, 64, 200, 200),
        # one sentence parsed online: inference, every step's output wanted
        _lstm("sentence_infer", "bf16", 153, 1, 200, 200, call="forward", wait=True),
        # a training step of a parser's stack, 64 sentences a minibatch
        _lstm("parser64", "bf16", 185, 64, 200, 200),
        # the same with twice the batch, dead writes skipped
        _lstm("parser128_push", "bf16", 185, 128, 200, 200, push_only=True),
        # a ragged batch of odd sizes: hold-padded sentences, row tiles and widths partly filled
        _lstm("ragged100", "bf16", 77, 100, 72, 104, ops="walk", probs=(0.5, 0.3, 0.2), ragged=True),
        # a corpus parsed in large batches: inference
        _lstm("parser512_infer", "bf16", 191, 512, 200, 200, call="forward"),
        # large-batch training of the same model
        _lstm("parser1024", "bf16", 195, 1024, 200, 200),
        # the three StackLSTMs of an arc-hybrid parser and its head, one training step
        dict(name="parser_step64", kind="parser", B=64, n=60, H=200, I=200, Ia=48, P=200),
        # a string-to-tree-decoder-like model: wide hidden state, ragged sentences
        _lstm("large256", "bf16", 256, 256, 512, 1024, ops="walk", probs=(0.5, 0.3, 0.2), ragged=True),
        # deep stacks, many instances, the loss on the final tops
        _lstm("stress4096", "bf16", 512, 4096, 256, 256, loss="top", ops="walk", probs=(0.6, 0.3, 0.1)),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _log8(rng, lo, hi):
    return 8 * max(1, _log(rng, lo / 8, hi / 8))


def draw(rng):
    """One more case of the listed ranges: the fp32 path up to parser64_fp32's sizes, the
    bf16 path at parser widths with up to 1024 instances, wide or very large batches up to
    stress4096's work, and parser steps."""
    which = rng.choice(("fp32", "parser", "parser", "wide", "step"))
    ops = rng.choice(("arc", "walk"))
    probs = rng.choice((_WALK, (0.5, 0.3, 0.2), (0.6, 0.3, 0.1)))
    more = dict(ops=ops, probs=probs, ragged=ops == "walk" and rng.random() < 0.5)
    if which == "fp32":
        return _lstm(None, "fp32", rng.randint(8, 185), _log(rng, 1, 64), _log(rng, 8, 200), _log(rng, 8, 200),
                     loss=rng.choice(("steps", "top")), **more)
    if which == "parser":
        call = rng.choice(("train", "train", "forward"))
        return _lstm(None, "bf16", rng.randint(16, 195), _log(rng, 1, 1024), _log8(rng, 16, 256), _log8(rng, 32, 256),
                     call=call, push_only=rng.random() < 0.25, loss=rng.choice(("steps", "top")), **more)
    if which == "wide":
        H, I = _log8(rng, 128, 1024), _log8(rng, 64, 512)
        T = rng.randint(64, 256)
        most = 0.6 * 512 * 4096 * 256 * 512 / (T * H * (I + H))
        return _lstm(None, "bf16", T, _log(rng, 96, max(128, min(4096, most))), I, H, push_only=rng.random() < 0.2,
                     loss=rng.choice(("steps", "top")), **more)
    return dict(kind="parser", B=_log(rng, 8, 128), n=rng.randint(12, 60), H=_log8(rng, 64, 256), I=_log8(rng, 32, 256),
                Ia=8 * rng.randint(1, 8), P=8 * rng.randint(8, 25))


# ------------------------------------------------------------------------------ inputs
def _walk(rng, T, B, probs, lengths):
    """Ops [T, B] drawn per step, no pop at depth 0 (its weight goes to the others), holds
    at and past an instance's length."""
    push, pop, hold = probs
    u = rng.random((T, B), dtype=np.float32)
    ops, depth = np.zeros((T, B), np.int8), np.zeros(B, np.int32)
    for t in range(T):
        op = np.where(u[t] < push, 1, np.where(u[t] < push + pop, -1, 0))
        op = np.where(depth == 0, np.where(u[t] < push / (push + hold), 1, 0), op)
        op = np.where(t < lengths, op, 0)
        ops[t] = op
        depth += op
    return ops


def _arc_standard(rng, T, B):
    """Ops [T, B] of random arc-standard derivations flattened to stack ops (Shift: push;
    Left-Arc: pop, pop, push; Right-Arc: pop), cut at T, holds past the end. Sentences have
    T / 18 to T / 3 tokens (10 to 60 at T = 185)."""
    n = rng.integers(max(1, T // 18), max(2, T // 3), B)
    ops, at = np.zeros((T, B), np.int8), np.zeros(B, np.int64)
    buf, stack = n.copy(), np.zeros(B, np.int64)
    cols = np.arange(B)

    def put(mask, op):
        m = mask & (at < T)
        ops[at[m], cols[m]] = op
        at[mask] += 1

    while True:
        live = ((buf > 0) | (stack > 1)) & (at < T)
        if not live.any():
            return ops
        n_valid = (buf > 0).astype(np.int64) + 2 * (stack >= 2)
        pick = (rng.random(B) * n_valid).astype(np.int64) + (buf == 0)  # 0 shift, 1 left, 2 right
        shift, left, right = live & (pick == 0), live & (pick == 1), live & (pick >= 2)
        put(shift, 1)
        put(left, -1)
        put(left, -1)
        put(left, 1)
        put(right, -1)
        buf -= shift
        stack += shift
        stack -= left | right


def _arc_hybrid(rng, B, n_max):
    """Random arc-hybrid derivations of n tokens (the first instance has n_max): n [B],
    transitions [2 n_max - 1, B] (0 shift, 1 left, 2 right; -1 past the end)."""
    n = rng.integers(max(1, n_max // 6), n_max + 1, B)
    n[0] = n_max
    T = 2 * n_max - 1
    tr, buf, stack = np.full((T, B), -1, np.int8), n.copy(), np.zeros(B, np.int64)
    for t in range(T):
        live = (buf > 0) | (stack > 1)
        can = np.stack([buf > 0, (stack >= 1) & (buf > 0), stack >= 2])
        pick = (rng.random(B) * can.sum(0)).astype(np.int64)
        op = np.argmax(np.cumsum(can, 0) == pick + 1, 0)
        tr[t] = np.where(live, op, -1)
        buf -= live & (op == 0)
        stack += np.where(live, np.where(op == 0, 1, -1), 0)
    return n, tr


class _Draw:
    """Seeded device tensors."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed))

    def normal(self, *shape, scale=1.0, dtype=torch.float32):
        return torch.randn(*shape, generator=self.g, device="cuda").mul_(scale).to(dtype)

    def uniform(self, *shape, r, dtype=torch.float32):
        return torch.rand(*shape, generator=self.g, device="cuda").mul_(2 * r).sub_(r).to(dtype)


def _tdtype(case):
    return torch.float32 if case["dtype"] == "fp32" else torch.bfloat16


def _lstm_inputs(case, seed):
    T, B, I, H, dt = case["T"], case["B"], case["I"], case["H"], _tdtype(case)
    rng = np.random.default_rng([int(seed), T, B, I, H])
    if case["ops"] == "arc":
        ops = _arc_standard(rng, T, B)
    else:
        lengths = rng.integers(max(1, T // 4), T + 1, B) if case["ragged"] else np.full(B, T)
        ops = _walk(rng, T, B, (case["push"], case["pop"], case["hold"]), lengths)
    d, r = _Draw(seed), 1.0 / math.sqrt(H)
    ins = dict(x=d.normal(T, B, I, dtype=dt), ops=torch.from_numpy(ops).cuda(), h0=d.uniform(B, H, r=0.5, dtype=dt),
               c0=d.uniform(B, H, r=0.5), W=d.uniform(I + H, 4 * H, r=r, dtype=dt), bias=d.uniform(4 * H, r=0.2))
    # the loss: a gradient for every step's output, or for the final top's h
    if case["call"] == "train":
        ins["d_top_h"] = d.normal(B, H) if case["loss"] == "top" else None
        ins["dy"] = d.normal(T, B, H) if case["loss"] == "steps" else None
    return ins


def _parser_inputs(case, seed):
    B, n_max, H, I, Ia, P = (case[k] for k in ("B", "n", "H", "I", "Ia", "P"))
    T, Tb, A, bf = 2 * n_max - 1, 3 * n_max - 1, 3, torch.bfloat16
    rng = np.random.default_rng([int(seed), B, n_max, H])
    n, tr = _arc_hybrid(rng, B, n_max)
    L = 2 * n - 1
    live = tr >= 0
    shift = tr == 0
    front = np.cumsum(shift, 0) - shift  # tokens shifted before each transition
    ops_s = np.where(live, np.where(shift, 1, -1), 0).astype(np.int8)
    ops_a = live.astype(np.int8)
    ops_b, tok_b = np.zeros((Tb, B), np.int8), np.full((Tb, B), -1)
    for b in range(B):
        ops_b[: n[b], b] = 1
        tok_b[: n[b], b] = np.arange(n[b] - 1, -1, -1)
        ops_b[n[b]: n[b] + L[b], b] = np.where(tr[: L[b], b] == 0, -1, 0)
    tok_s = np.where(live & (front < n), front, -1)
    d = _Draw(seed)
    rep, emb = d.normal(n_max, B, I, dtype=bf), d.normal(A, Ia, dtype=bf)
    cols = torch.arange(B, device="cuda")

    def tokens(tok):
        tok = torch.from_numpy(tok).cuda()
        return torch.where((tok >= 0)[..., None], rep[tok.clamp(min=0), cols], torch.zeros((), dtype=bf, device="cuda"))

    gold = torch.from_numpy(tr).cuda()
    x_a = torch.where((gold >= 0)[..., None], emb[gold.long().clamp(min=0)], torch.zeros((), dtype=bf, device="cuda"))
    members = {}
    for k, ops, x in (("stack", ops_s, tokens(tok_s)), ("buffer", ops_b, tokens(tok_b)), ("action", ops_a, x_a)):
        members[k] = dict(x=x.contiguous(), ops=torch.from_numpy(ops).cuda(), h0=d.uniform(B, H, r=0.5, dtype=bf),
                          c0=d.uniform(B, H, r=0.5), W=d.uniform(x.shape[2] + H, 4 * H, r=1.0 / math.sqrt(H), dtype=bf),
                          bias=d.uniform(4 * H, r=0.2))
    head = dict(n=torch.from_numpy(n.astype(np.int32)).cuda(), L=torch.from_numpy(L.astype(np.int32)).cuda(), gold=gold,
                Wp=d.uniform(P, 3 * H, r=1.0 / math.sqrt(3 * H), dtype=bf), dp=d.uniform(P, r=1.0),
                Wz=d.uniform(A, P, r=1.0 / math.sqrt(P)), q=d.uniform(A, r=0.1))
    return members, head


def _empty(*shape, dtype=torch.float32):
    return torch.empty(*shape, dtype=dtype, device="cuda")


def _grads(T, B, I, H):
    return dict(dx=_empty(T, B, I), dh0=_empty(B, H), dc0=_empty(B, H), dW=_empty(I + H, 4 * H), dbias=_empty(4 * H))


def prepare(case, seed):
    if case["kind"] == "parser":
        members, hin = _parser_inputs(case, seed)
        B, H, P, A = case["B"], case["H"], case["P"], 3
        T, Tb = 2 * case["n"] - 1, 3 * case["n"] - 1
        hds, outs = {}, {}
        for k, m in members.items():
            (t, _, i), st = m["x"].shape, torch.cuda.Stream()
            hd = bd.stacklstm_create(t, B, i, H, bd.SL_BF16, 0, st)
            bd.stacklstm_set_async(hd, True)
            hds[k] = (hd, st)
            outs[k] = dict(p_final=_empty(B, dtype=torch.int32), y=_empty(t, B, H, dtype=torch.bfloat16),
                           **_grads(t, B, i, H))
        hout = dict(loss_rows=_empty(T, B), dy_stack=_empty(T, B, H), dy_buffer=_empty(Tb, B, H),
                    dy_action=_empty(T, B, H), dWp=_empty(P, 3 * H), ddp=_empty(P), dWz=_empty(A, P), dq=_empty(A))
        head = bd.stacklstm_head_create(T, Tb, B, H, P, A)
        return dict(case=case, ps=dict(hds=hds, head=head, hin=hin, hout=hout, ins=members, outs=outs))
    T, B, I, H = case["T"], case["B"], case["I"], case["H"]
    hd = bd.stacklstm_create(T, B, I, H, bd.SL_FP32 if case["dtype"] == "fp32" else bd.SL_BF16)
    if not case["wait"]:
        bd.stacklstm_set_async(hd, True)
    if case["push_only"]:
        bd.stacklstm_set_mode(hd, bd.SL_MODE_PUSH_ONLY)
    out = dict(p_final=_empty(B, dtype=torch.int32))
    if case["call"] == "forward" or case["loss"] == "steps":
        out["y"] = _empty(T, B, H, dtype=_tdtype(case))
    if case["call"] == "train":
        out.update(_grads(T, B, I, H))
    return dict(case=case, hd=hd, ins=_lstm_inputs(case, seed), out=out)


def run(state):
    case = state["case"]
    if case["kind"] == "parser":
        runner.parser_step(state["ps"])
        return dict(state["ps"]["outs"], head=state["ps"]["hout"])
    ins, out = state["ins"], state["out"]
    if case["call"] == "train":
        runner.forward_backward(state["hd"], ins, out)
    else:
        bd.stacklstm_forward(state["hd"], ins["x"], ins["ops"], ins["h0"], ins["c0"], ins["W"], ins["bias"],
                             p_final=out["p_final"], y=out["y"])
    return out


# -------------------------------------------------------------------------------- work
def _lstm_work(T, B, I, H, es, train, y, dy):
    """Inputs and outputs once; 2 flops a multiply-add of the gate contraction, and twice as
    many again for the input, state and weight gradients."""
    R, w = T * B, (I + H) * 4 * H
    by = es * (R * I + B * H + w) + R + 4 * (B * H + 4 * H) + 4 * B + (es * R * H if y else 0)
    if train:
        by += 4 * (R * I + 2 * B * H + w + 4 * H) + 4 * (R * H if dy else B * H)
    return by, 2 * R * w * (3 if train else 1)


def work(case):
    if case["kind"] == "parser":
        B, H, P, n = case["B"], case["H"], case["P"], case["n"]
        T, Tb = 2 * n - 1, 3 * n - 1
        by = fl = 0
        for t, i in ((T, case["I"]), (Tb, case["I"]), (T, case["Ia"])):
            b, f = _lstm_work(t, B, i, H, 2, True, True, False)
            by, fl = by + b + 4 * t * B * H, fl + f  # y and the head's gradient of it are outputs
        by += T * B * 5 + 2 * 3 * H * P + 4 * (3 * H * P + 8 * P + 6)
        return {"bytes": by, "flops": fl + 6 * T * B * P * (3 * H + 3)}
    T, B, I, H = case["T"], case["B"], case["I"], case["H"]
    train = case["call"] == "train"
    y = case["call"] == "forward" or case["loss"] == "steps"
    by, fl = _lstm_work(T, B, I, H, 4 if case["dtype"] == "fp32" else 2, train, y, case["loss"] == "steps")
    if case["push_only"]:
        # only the pushes need computing: a derivation's share of them, or the walk's
        fl = int(fl * (0.28 if case["ops"] == "arc" else case["push"] * (0.6 if case["ragged"] else 1.0)))
    return {"bytes": by, "flops": fl}


# --------------------------------------------------------------------------- tolerance
def tolerance(case):
    """About four times what each path shows against 64-bit arithmetic on these inputs."""
    if case["kind"] == "parser":
        # the head's ReLU: a state within bf16 rounding of zero passes its gradient on one side
        # and not on the other, so single rows of the gradients differ
        return {"rel": 3e-2, "max": 0.99}
    if case["dtype"] == "fp32":
        return {"rel": 4e-6, "max": 1e-4}
    # bf16 operands and states: rounding of 2^-9 a value, through the recurrence (0.3e-2 seen)
    return {"rel": 1e-2, "max": 0.6}


# ------------------------------------------------------------------------------- exact
def _tops(ops):
    """src [T + 1, B] (0: the initial state, t + 1: the state step t wrote) and the final
    pointers, by replaying the ops on a table of slots."""
    ops = ops.cpu().numpy().astype(np.int64)
    T, B = ops.shape
    cols, p, tags, src = np.arange(B), np.zeros(B, np.int64), np.zeros((T + 2, B), np.int64), np.zeros((T + 1, B), np.int64)
    for t in range(T):
        src[t] = tags[p, cols]
        tags[p + 1, cols] = t + 1
        p = p + ops[t]
    src[T] = tags[p, cols]
    return torch.from_numpy(src).cuda(), torch.from_numpy(p.astype(np.int32)).cuda()


def _forward64(ins):
    x, W = ins["x"].double(), ins["W"].double()
    T, B, I = x.shape
    H = W.shape[1] // 4
    src, p_final = _tops(ins["ops"])
    h, c = (torch.empty(T + 1, B, H, dtype=torch.float64, device="cuda") for _ in range(2))
    h[0], c[0] = ins["h0"].double(), ins["c0"].double()
    gates, cols = torch.empty(T, B, 4 * H, dtype=torch.float64, device="cuda"), torch.arange(B, device="cuda")
    for t in range(T):
        z = torch.addmm(ins["bias"].double(), x[t], W[:I]).addmm_(h[src[t], cols], W[I:])
        i, f, g, o = z.view(B, 4, H).unbind(1)
        i, f, g, o = i.sigmoid(), f.sigmoid(), g.tanh(), o.sigmoid()
        torch.stack((i, f, g, o), 1, out=gates[t].view(B, 4, H))
        c[t + 1] = f * c[src[t], cols] + i * g
        h[t + 1] = o * c[t + 1].tanh()
    y = h[src[1:], cols]
    return dict(x=x, W=W, src=src, cols=cols, h=h, c=c, gates=gates, y=y, p_final=p_final)


def _backward64(s, d_top_h, dy):
    x, W, src, cols, h, c, gates = (s[k] for k in ("x", "W", "src", "cols", "h", "c", "gates"))
    T, B, I = x.shape
    H = W.shape[1] // 4
    dh, dc = torch.zeros_like(h), torch.zeros_like(c)
    if d_top_h is not None:
        dh[src[T], cols] += d_top_h.double()
    if dy is not None:
        for t in range(T):
            dh[src[t + 1], cols] += dy[t].double()
    dz, Wh_t, dW, db = torch.empty_like(gates), W[I:].t().contiguous(), torch.zeros_like(W), 0
    for t in range(T - 1, -1, -1):
        i, f, g, o = gates[t].view(B, 4, H).unbind(1)
        tc = c[t + 1].tanh()
        dct = dc[t + 1] + dh[t + 1] * o * (1 - tc * tc)
        cr = c[src[t], cols]
        torch.stack((dct * g * i * (1 - i), dct * cr * f * (1 - f), dct * i * (1 - g * g), dh[t + 1] * tc * o * (1 - o)), 1,
                    out=dz[t].view(B, 4, H))
        dc[src[t], cols] += dct * f
        dh[src[t], cols] += dz[t] @ Wh_t
    step = max(1, (1 << 18) // B)  # a few hundred thousand rows at a time
    for t in range(0, T, step):
        rows = dz[t:t + step].reshape(-1, 4 * H)
        n = rows.shape[0] // B
        dW[:I].addmm_(x[t:t + n].reshape(-1, I).t(), rows)
        dW[I:].addmm_(h[src[t:t + n], cols].reshape(-1, H).t(), rows)
        db = db + rows.sum(0)
    return dict(dx=dz @ W[:I].t(), dh0=dh[0], dc0=dc[0], dW=dW, dbias=db)


def _head64(m, hin):
    y = {k: v["y"] for k, v in m.items()}
    T, B, H = y["stack"].shape
    n, L = hin["n"].long(), hin["L"].long()
    k, cols = torch.arange(T, device="cuda")[:, None], torch.arange(B, device="cuda")
    live = k < L
    at_b = (n - 1 + k).clamp(max=y["buffer"].shape[0] - 1)
    tops = [torch.cat((m["stack"]["h"][:1], y["stack"][:-1])), y["buffer"][at_b, cols],
            torch.cat((m["action"]["h"][:1], y["action"][:-1]))]
    u = torch.where(live[..., None], torch.cat(tops, 2), torch.zeros((), dtype=torch.float64, device="cuda"))
    Wp, Wz = hin["Wp"].double(), hin["Wz"].double()
    p = (u @ Wp.t() + hin["dp"].double()).relu()
    z = p @ Wz.t() + hin["q"].double()
    gold, lse = hin["gold"].long().clamp(min=0), z.logsumexp(2)
    rows = (lse - z.gather(2, gold[..., None])[..., 0]) * live
    dz = z.softmax(2)
    dz.scatter_add_(2, gold[..., None], -torch.ones_like(dz[..., :1]))
    dz *= live[..., None]
    dp = (dz @ Wz) * (p > 0)
    du = dp @ Wp
    out = dict(loss_rows=rows, dWp=dp.flatten(0, 1).t() @ u.flatten(0, 1), ddp=dp.sum((0, 1)),
               dWz=dz.flatten(0, 1).t() @ p.flatten(0, 1), dq=dz.sum((0, 1)))
    dys = {q: torch.zeros_like(y[q]) for q in y}
    dys["stack"][:-1], dys["action"][:-1] = du[1:, :, :H], du[1:, :, 2 * H:]
    # rows past an instance's transitions carry zero, so where they clamp to makes no difference
    dys["buffer"].index_put_((at_b, cols.expand(T, B)), du[..., H:2 * H], accumulate=True)
    out.update({"dy_" + q: v for q, v in dys.items()})
    return out, du[0, :, :H], du[0, :, 2 * H:]


def exact(case, seed):
    if case["kind"] == "parser":
        members, hin = _parser_inputs(case, seed)
        fwd = {k: _forward64(m) for k, m in members.items()}
        head, dh_s, dh_a = _head64(fwd, hin)
        out = {k: dict(p_final=f["p_final"], y=f["y"], **_backward64(f, None, head["dy_" + k])) for k, f in fwd.items()}
        out["stack"]["dh0"] += dh_s
        out["action"]["dh0"] += dh_a
        return dict(out, head=head)
    ins = _lstm_inputs(case, seed)
    f = _forward64(ins)
    out = dict(p_final=f["p_final"])
    if case["call"] == "forward" or case["loss"] == "steps":
        out["y"] = f["y"]
    if case["call"] == "train":
        out.update(_backward64(f, ins["d_top_h"], ins["dy"]))
    return out
