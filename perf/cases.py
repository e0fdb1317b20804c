"""What a student update asks of this library, as measured cases.

Every case goes through paper_2609_36246_gb300.binding, as a training program does: sequences are
a student prefix followed by a teacher continuation, and the masked rows are those that predict
continuation tokens.  Ids, hidden rows and LM heads are drawn on the GPU from the seed.  Hidden
rows are RMS-normalised Gaussians that lean towards the LM-head row of the token they predict, by
a different amount for each row, so that target probabilities run from 1/V up to nearly 1; the
teacher leans towards the same tokens, as two models that mostly agree do.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2609_36246_gb300 import binding as B

W_STD = 0.02  # standard deviation of the LM-head weights (synth.py)
LEAN = 0.35   # most of a hidden row that points at its target's LM-head row

DEFAULTS = dict(op="train", seqs=1, prefix=1, cont=1, ragged=False, d=4096, d_t=0, V=151936, K=16,
                grad="bf16", tau=1.0, reduction="sum", direction="reverse", flags=1.0)


def listed():
    c = lambda name, **kw: dict(DEFAULTS, name=name, **kw)
    return [
        # one optimiser step's packing: 64 prompts x 4 rollouts, a student prefix of about 4096
        # tokens and a teacher continuation of about 1024, lengths ragged
        c("pack_step", op="pack", seqs=256, prefix=4096, cont=1024, ragged=True),
        # multi-turn packing of a variable-length batch: only the teacher's actions carry the loss
        c("pack_turns", op="pack_turns", seqs=64, prefix=4000, cont=4257, ragged=True, flags=0.4),
        # the smallest training step (4 x 128 tokens, d = 256, V = 4096): launches and host time
        c("train_tiny", op="train", seqs=4, prefix=64, cont=64, ragged=True, d=256, V=4096),
        # autograd op on two short continuations: a small micro-batch over a full vocabulary
        c("autograd_short", op="autograd", seqs=2, prefix=700, cont=150, ragged=True, d=2048),
        # one rollout: prefix cut at student token 4096, 1024-token teacher continuation
        c("train_rollout", op="train", seqs=1, prefix=4096, cont=1024),
        # the training step of a micro-batch of 8 x 4096 tokens with ragged cuts
        c("train_batch", op="train", seqs=8, prefix=2008, cont=2088, ragged=True),
        # forward, then a backward whose loss gradient is known late: mean reduction, fp32
        # gradients, a temperature, an odd vocabulary
        c("two_call", op="two_call", seqs=3, prefix=1500, cont=613, ragged=True, d=2560, V=100003,
          grad="f32", tau=0.9, reduction="mean"),
        # scoring one short continuation: one pass over the LM head, few rows
        c("score_short", op="score", seqs=1, prefix=512, cont=96),
        # forward scoring of a batch: 2 x (4096 + 4096) tokens, d = 2048
        c("score_batch", op="score", seqs=2, prefix=4096, cont=4096, d=2048),
        # distillation by the full-vocabulary reverse KL, gradient for the student: 4 rollouts
        c("kl_grad", op="kl_grad", seqs=4, prefix=512, cont=1024, d=4096, d_t=5120),
        # OPD's per-token statistics of one long rollout
        c("opd_stats", op="opd", seqs=1, prefix=100, cont=2900, d=4096, d_t=5120),
        # the top-16 KL training step (teacher sweep, then the student's forward and backward)
        c("topk_kl_step", op="topk_kl", seqs=2, prefix=512, cont=1024, d=4096, d_t=5120),
    ]


OPS = ("train", "train", "train", "autograd", "two_call", "slab", "score", "score", "topk", "kl",
       "kl_grad", "kl_grad", "opd", "topk_kl", "pack", "pack_turns")


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(OPS)
    c = dict(DEFAULTS, op=op, ragged=rng.random() < 0.7, tau=rng.choice((1.0, 1.0, 0.8, 1.1)),
             reduction=rng.choice(("sum", "sum", "mean")), grad=rng.choice(("bf16", "bf16", "f32")),
             direction=rng.choice(("reverse", "reverse", "forward")), K=rng.choice((16, 16, 8, 1)))
    if op.startswith("pack"):
        c.update(seqs=_log_int(rng, 1, 256), prefix=_log_int(rng, 16, 4096),
                 cont=_log_int(rng, 16, 2048), flags=rng.uniform(0.1, 0.9))
        return c
    c.update(d=8 * _log_int(rng, 32, 512), V=_log_int(rng, 4096, 151936),
             seqs=_log_int(rng, 1, 8), prefix=_log_int(rng, 16, 2048))
    if op in ("kl", "kl_grad", "opd", "topk_kl"):
        c["d_t"] = 8 * _log_int(rng, 32, 640)
    # masked rows over the range of a micro-batch, within the largest listed case's work
    most = 5e13 / (6.0 * c["V"] * max(c["d"], c["d_t"]))
    rows = _log_int(rng, 24, max(32, min(16384, int(most))))
    c["seqs"] = min(c["seqs"], max(1, rows // 8))
    c["cont"] = max(8, rows // c["seqs"])
    return c


def _lengths(c):
    """Prefix and continuation lengths of a case, the same for every seed."""
    rng = random.Random("%d %d %d" % (c["seqs"], c["prefix"], c["cont"]))
    part = lambda n: max(1, int(n * rng.uniform(0.5, 1.5))) if c["ragged"] else n
    return ([part(c["prefix"]) for _ in range(c["seqs"])], [part(c["cont"]) for _ in range(c["seqs"])])


def _sizes(c):
    p, k = _lengths(c)
    return sum(p) + sum(k), sum(k)


def _layout(c):
    """Packed starts, cuts and the masked rows (those before a continuation token), as numpy."""
    p, k = _lengths(c)
    starts = np.concatenate([[0], np.cumsum(np.add(p, k))]).astype(np.int64)
    cuts = starts[:-1] + np.array(p)
    rows = np.concatenate([np.arange(a - 1, a + n - 1) for a, n in zip(cuts, k)])
    return p, k, starts, cuts, rows


def _csr(n):
    return torch.tensor(np.concatenate([[0], np.cumsum(n)]).astype(np.int32), device="cuda")


def _ids(c, gen):
    p, k = _lengths(c)
    draw_ids = lambda n: torch.randint(0, c["V"], (n,), generator=gen, device="cuda", dtype=torch.int32)
    return dict(prefix_ids=draw_ids(sum(p)), prefix_off=_csr(p), cont_ids=draw_ids(sum(k)),
                cont_off=_csr(k))


def _packed(c, s):
    """The packed ids and targets of the drawn batch, in plain torch."""
    p, k, starts, _, _ = _layout(c)
    T = int(starts[-1])
    pre, con = s["prefix_ids"].split(p), s["cont_ids"].split(k)
    ids = torch.cat([x for pair in zip(pre, con) for x in pair])
    targets = torch.cat([ids[1:], ids.new_full((1,), -1)])
    targets[torch.tensor(starts[1:] - 1, device="cuda")] = -1
    return T, ids, targets


def _head(V, d, gen):
    return (torch.randn(V, d, generator=gen, device="cuda") * W_STD).to(torch.bfloat16)


def _hidden(T, W, targets, gen):
    h = torch.randn(T, W.shape[1], generator=gen, device="cuda")
    lean = torch.rand(T, 1, generator=gen, device="cuda") * LEAN
    y = targets.clamp(min=0).long()
    for a in range(0, T, 8192):
        h[a:a + 8192] += lean[a:a + 8192] / W_STD * W[y[a:a + 8192]].float()
    h *= (h.square().mean(1, keepdim=True) + 1e-6).rsqrt()
    return h.to(torch.bfloat16)


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = dict(c=c, **_ids(c, gen))
    T, n = _sizes(c)
    s["T"], s["n"] = T, n
    if c["op"] == "pack_turns":
        s["n"] = max(1, int(n * c["flags"]))
        s["cont_loss"] = torch.zeros(n, dtype=torch.uint8, device="cuda")
        s["cont_loss"][torch.randperm(n, generator=gen, device="cuda")[: s["n"]]] = 1
    if c["op"].startswith("pack"):
        return s
    _, _, targets = _packed(c, s)
    s["targets"] = targets
    s["rows"] = torch.tensor(_layout(c)[4].astype(np.int32), device="cuda")
    s["n_rows"] = torch.full((1,), n, dtype=torch.int32, device="cuda")
    s["W"] = _head(c["V"], c["d"], gen)
    s["hidden"] = _hidden(T, s["W"], targets, gen)
    s["dtype"] = torch.float32 if c["grad"] == "f32" else torch.bfloat16
    if c["op"] in ("kl", "kl_grad", "opd", "topk_kl"):
        s["W_t"] = _head(c["V"], c["d_t"], gen)
        s["h_t"] = _hidden(T, s["W_t"], targets, gen)
        s["weight"] = torch.rand(T, generator=gen, device="cuda") + 0.5  # per-token loss weights
    s["grad_loss"] = torch.full((1,), 0.75, dtype=torch.float32, device="cuda")
    if c["op"] == "autograd":
        s["hidden"].requires_grad_(True)
        s["W"].requires_grad_(True)
    return s


PACKED = ("ids", "targets", "loss_mask", "cu_seqlens", "cut_offsets", "n_rows", "dev_status")


def run(state):
    s, c = state, state["c"]
    op, tau = c["op"], 1.0 / c["tau"]
    if op in ("pack", "pack_turns", "train", "slab", "score"):
        csr = (s["prefix_ids"], s["prefix_off"], s["cont_ids"], s["cont_off"])
        if op == "pack_turns":
            pk = B.olive_splice_pack_masked(*csr, s["cont_loss"], c["V"], s["T"])
        else:
            pk = B.olive_splice_pack(*csr, c["V"], s["T"])
        if op.startswith("pack"):
            # the call defines the first n_rows entries of rows
            return dict({k: pk[k] for k in PACKED}, rows=pk["rows"][: s["n"]])
        rows, n_rows, targets, h, W = pk["rows"], pk["n_rows"], pk["targets"], s["hidden"], s["W"]
        if op == "score":
            return B.olive_token_logprob_fwd(h, W, targets, rows, n_rows, tau, c["reduction"])
        return B.olive_token_loss_fwd_bwd(h, W, targets, rows, n_rows, s["grad_loss"], tau,
                                          c["reduction"], s["dtype"], slab=op == "slab")
    h, W, rows, n_rows = s["hidden"], s["W"], s["rows"], s["n_rows"]
    if op == "autograd":
        loss = B.fused_lmhead_ce(h, W, s["targets"], rows, n_rows, tau, c["reduction"])
        d_h, d_W = torch.autograd.grad(loss * s["grad_loss"][0], (h, W))
        return loss.detach(), d_h, d_W
    if op == "two_call":
        logp, lse, loss = B.olive_token_logprob_fwd(h, W, s["targets"], rows, n_rows, tau,
                                                    c["reduction"])
        d_h, d_W = B.olive_token_loss_bwd(h, W, s["targets"], rows, n_rows, lse, s["grad_loss"], tau,
                                          c["reduction"], s["dtype"])
        return logp, lse, loss, d_h, d_W
    if op == "topk":
        return B.olive_token_topk_fwd(h, W, rows, n_rows, c["K"], tau)
    if op == "kl":
        return B.olive_token_divergence(h, W, s["h_t"], s["W_t"], rows, n_rows, tau,
                                        c["direction"])[0]
    if op == "kl_grad":
        return B.olive_token_divergence(h, W, s["h_t"], s["W_t"], rows, n_rows, tau, c["direction"],
                                        s["weight"], s["dtype"])
    if op == "opd":
        return B.olive_opd_token_stats(h, W, s["h_t"], s["W_t"], rows, n_rows, c["K"], tau,
                                       c["direction"])
    t_lse, t_ent, t_logp, t_ids = B.olive_token_topk_fwd(s["h_t"], s["W_t"], rows, n_rows, c["K"], tau)
    out = B.olive_topk_kl_fwd_bwd(h, W, s["h_t"], s["W_t"], rows, n_rows, c["K"], t_lse, s["weight"],
                                  t_ids, tau, s["dtype"])
    return dict(out, t_lse=t_lse, t_entropy=t_ent, t_topk_logp=t_logp, t_topk_ids=t_ids)


def work(case):
    """Inputs read once, outputs written once, products computed once (masked rows only)."""
    c = case
    T, n = _sizes(c)
    if c["op"].startswith("pack"):
        ids = 4 * T + 8 * (c["seqs"] + 1) + (n if c["op"] == "pack_turns" else 0)
        marked = n * c["flags"] if c["op"] == "pack_turns" else n
        return dict(bytes=ids + 9 * T + 8 * c["seqs"] + 4 * marked, flops=0)
    d, dt, V, K = c["d"], c["d_t"], c["V"], c["K"]
    e = 4 if c["grad"] == "f32" else 2
    one, teacher = 2.0 * n * d * V, 2.0 * n * dt * V
    head, rows_in, grads = 2.0 * V * d, 2.0 * n * d + 8 * n, e * (T * d + V * d)
    both = head + rows_in + 2.0 * V * dt + 2.0 * n * dt
    if c["op"] in ("train", "slab", "autograd", "two_call"):
        return dict(bytes=head + rows_in + grads + 8 * T, flops=3 * one)
    if c["op"] == "score":
        return dict(bytes=head + rows_in + 8 * T, flops=one)
    if c["op"] == "topk":
        return dict(bytes=head + rows_in + 8 * T * (1 + K), flops=one)
    if c["op"] == "kl":
        return dict(bytes=both + 4 * T, flops=one + teacher)
    if c["op"] == "kl_grad":
        return dict(bytes=both + 4 * T + e * T * d, flops=2 * one + teacher)
    if c["op"] == "opd":
        return dict(bytes=both + 4 * T * (6 + 3 * K), flops=one + teacher)
    return dict(bytes=both + 4 * T * (6 + 5 * K) + grads, flops=3 * one + teacher)


def tolerance(case):
    """The largest relative error over a call's outputs that rounding explains."""
    op = case["op"]
    if op.startswith("pack"):
        return "exact"
    if op in ("score", "kl", "topk"):
        # fp32 sums of exact bf16 products: up to 9e-6 from 64 bits; ids: neighbours in a top list
        # closer than the rounding of such a sum swap places
        return dict(rel=4e-5, max=1e-3, differ=2e-3)
    if op == "opd":
        # the teacher's log-probs at swapped ids: 1.3e-3 from 64 bits
        return dict(rel=5e-3, max=0.9, differ=2e-3)
    # gradients: the logit gradient is an operand in bf16 (2^-9), and so may the result be: up to
    # 3e-3 from 64 bits
    return dict(rel=1e-2, max=0.9 if op == "topk_kl" else 0.3, differ=2e-3)


def _logits(s, h, W, r, tau):
    return h[r].double() @ W.t() / tau


def exact(case, seed):
    c = case
    T, n = _sizes(c)
    if c["op"].startswith("pack"):
        return _exact_pack(c, seed)
    if work(c)["flops"] > 9e12:  # a few seconds of this GPU's fp64 rate
        return None
    s = prepare(dict(c), seed)
    h, W = s["hidden"].detach(), s["W"].detach().double()
    rows, tau, K, op, V = s["rows"].long(), c["tau"], c["K"], c["op"], c["V"]
    teacher = op in ("kl", "kl_grad", "opd", "topk_kl")
    W_t = s["W_t"].double() if teacher else None
    zeros = lambda *shape: torch.zeros(*shape, dtype=torch.float64, device="cuda")
    whole = lambda *shape: torch.full(shape, -1, dtype=torch.int32, device="cuda")
    logp, lse, kl, ent, t_lse, t_ent, kl_k, over = (zeros(T) for _ in range(8))
    top_v, t_at_s, t_top_v = zeros(T, K), zeros(T, K), zeros(T, K)
    top_i, t_top_i = whole(T, K), whole(T, K)
    gradient = op in ("train", "slab", "autograd", "two_call", "kl_grad", "topk_kl")
    d_h, d_W = zeros(T, c["d"]) if gradient else None, None
    if gradient and op != "kl_grad":
        d_W = zeros(V, c["d"])
    scale = 0.75 / (n if c["reduction"] == "mean" else 1) / tau
    for a in range(0, n, 256):
        r = rows[a:a + 256]
        z = _logits(s, h, W, r, tau)
        lse[r] = z.logsumexp(1)
        l = z - lse[r, None]
        p = l.exp()
        if teacher:
            zt = _logits(s, s["h_t"], W_t, r, tau)
            t_lse[r] = zt.logsumexp(1)
            lt = zt - t_lse[r, None]
            pt = lt.exp()
            w = s["weight"].double()[r, None]
        G = None
        if not teacher and op != "topk":
            y = s["targets"][r].long()[:, None]
            logp[r] = l.gather(1, y)[:, 0]
            if gradient:
                G = p * scale
                G.scatter_add_(1, y, torch.full_like(y, -scale, dtype=torch.float64))
        if op in ("topk", "opd", "topk_kl"):
            ent[r] = -(p * l).sum(1)
            v, i = l.topk(K, 1)
            top_v[r], top_i[r] = v, i.int()
        if op in ("kl", "kl_grad", "opd"):
            back = c["direction"] == "reverse"
            kl[r] = (p * (l - lt)).sum(1) if back else (pt * (lt - l)).sum(1)
            if gradient:
                G = w / tau * (p * (l - lt - kl[r, None]) if back else p - pt)
        if op in ("opd", "topk_kl"):
            tv, ti = lt.topk(K, 1)
            t_top_v[r], t_top_i[r] = tv, ti.int()
            t_ent[r] = -(pt * lt).sum(1)
            q = lt.gather(1, i)
            t_at_s[r] = q
            over[r] = (i[:, :, None] == ti[:, None, :]).any(2).double().mean(1)
            kl_k[r] = (v.exp() * (v - q)).sum(1)
            if gradient:
                mass = v.exp().sum(1)
                G = p * -(kl_k[r] + mass)[:, None]
                G.scatter_add_(1, i, v.exp() * (v - q + 1))
                G *= w / tau
        if G is not None:
            d_h[r] = G @ W
            if d_W is not None:
                d_W += G.t() @ h[r].double()
    loss = -logp.sum().reshape(1) / (n if c["reduction"] == "mean" else 1)
    if op == "score":
        return logp, lse, loss
    if op == "autograd":
        return loss[0], d_h, d_W
    if op in ("train", "slab", "two_call"):
        return logp, lse, loss, d_h, d_W
    if op == "topk":
        return lse, ent, top_v, top_i
    if op == "kl":
        return kl
    if op == "kl_grad":
        return kl, d_h
    if op == "opd":
        return dict(kl=kl, s_lse=lse, t_lse=t_lse, s_entropy=ent, s_topk_logp=top_v, s_topk_ids=top_i,
                    t_logp_s=t_at_s, overlap=over, kl_topk=kl_k)
    return dict(s_lse=lse, s_ids=top_i, s_logp=top_v, t_logp_s=t_at_s, kl_topk=kl_k, overlap=over,
                d_h_s=d_h, d_W_s=d_W, t_lse=t_lse, t_entropy=t_ent, t_topk_logp=t_top_v,
                t_topk_ids=t_top_i)


def _exact_pack(c, seed):
    s = prepare(dict(c), seed)
    p, k, starts, cuts, rows = _layout(c)
    T, ids, targets = _packed(c, s)
    if c["op"] == "pack_turns":
        rows = rows[s["cont_loss"].cpu().numpy() != 0]
    mask = np.zeros(T, np.uint8)
    mask[rows] = 1
    i32 = lambda x: torch.tensor(np.asarray(x).astype(np.int32))
    return dict(ids=ids, targets=targets, loss_mask=torch.tensor(mask), cu_seqlens=i32(starts),
                cut_offsets=i32(cuts), n_rows=i32([len(rows)]), dev_status=i32([0]), rows=i32(rows))
