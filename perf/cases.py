"""The verification, drafting and decoding work that users of this library have it do, as measurable cases.

A case names an entry point and the sizes of one call.  ``kind`` is one of

  block, token, greedy        bv_verify (Algorithm 2), tv_verify (Algorithm 1), gbv_verify (Algorithm 4) on logits
  block_lse, token_lse        the same with the draft rows' log-normalisers handed over from the drafting step
  block_probs, token_probs    on probabilities instead of logits
  block_ex                    Algorithm 2 with its intermediates (acceptance weights, residual masses, normalisers)
  block_host, token_host      on pinned host buffers, copies included
  sample                      bv_sample_draft: one token and the log-normaliser for each of B rows of draft logits
  loop                        specdec.run: ``iters`` iterations of the decoding loop on two last-token model tables

``B`` sequences (rows for "sample") of ``gamma`` drafted tokens over a vocabulary of ``V`` tokens, ``dtype`` the
storage type of the logits, ``temperature``; ``sigma_d`` is the draft's noise against the target (0.1: nearly every
token is accepted, 1: one or two, 3: hardly any); ``head`` how peaked the target rows are (see _rows); ``masked``
rows keep about a tenth of their vocabulary, as nucleus or top-k sampling leaves them.
"""
import math

import torch

from paper_2403_10444_b200 import binding as bv
from paper_2403_10444_b200 import specdec

VERIFY = {"block": bv.bv_verify, "token": bv.tv_verify, "greedy": bv.gbv_verify, "block_ex": bv.bv_verify_ex}
VERIFY_LSE = {"block_lse": bv.bv_verify_lse, "token_lse": bv.tv_verify_lse}
VERIFY_PROBS = {"block_probs": bv.bv_verify_probs, "token_probs": bv.tv_verify_probs}
VERIFY_HOST = {"block_host": bv.bv_verify_host, "token_host": bv.tv_verify_host}
ANY_V = ("block", "token", "block_ex", "block_host", "token_host")      # the others take rows of whole 16-byte vectors


def _case(name, kind, B, gamma, V, dtype="bf16", temperature=1.0, sigma_d=1.0, head="zipf", masked=False, iters=0):
    c = dict(kind=kind, B=B, gamma=gamma, V=V, dtype=dtype, temperature=temperature, sigma_d=sigma_d, head=head,
             masked=masked, iters=iters)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one interactive request: the smallest call, all latency
        _case("block_1", "block", 1, 8, 152064, temperature=0.8),
        # a handful of requests, fp32 logits of a 32000-token vocabulary with a few strong tokens per row
        _case("block_8_f32", "block", 8, 8, 32000, dtype="f32", head="boost"),
        # a server's ordinary batch
        _case("block_64", "block", 64, 8, 128256, temperature=0.8, sigma_d=0.7),
        # a full batch over a large vocabulary: the library's headline workload
        _case("block_256", "block", 256, 8, 256000, sigma_d=1.5, head="broad"),
        # a well matched draft with long blocks: nearly every position can be the selected one
        _case("block_96_close", "block", 96, 12, 152064, temperature=0.8, sigma_d=0.1),
        # a vocabulary that is no multiple of anything, as tokenizers leave it: rows at every alignment
        _case("block_24_odd", "block", 24, 5, 50257, sigma_d=0.8),
        # the baseline algorithm on a full batch
        _case("token_256", "token", 256, 8, 152064, temperature=0.8),
        # drafted by this library, so the draft rows' normalisers come along
        _case("lse_64", "block_lse", 64, 8, 128256, temperature=0.8, sigma_d=0.7),
        # a serving stack that hands over softmax outputs
        _case("probs_64", "block_probs", 64, 8, 128256, temperature=0.8, sigma_d=0.7),
        # one drafting step of a full batch
        _case("sample_256", "sample", 256, 1, 128256, temperature=0.8, sigma_d=0.7),
        # the whole loop: draft, look up, verify, extend
        _case("loop_128", "loop", 128, 5, 16384, iters=8),
        # logits that live on the host
        _case("host_8_f32", "block_host", 8, 8, 32000, dtype="f32", head="boost"),
    ]


KINDS = (("block", 8), ("token", 4), ("block_lse", 2), ("token_lse", 1), ("block_probs", 1), ("token_probs", 1), ("greedy", 1),
         ("block_ex", 1), ("sample", 3), ("loop", 1), ("block_host", 1), ("token_host", 1))
VOCABULARIES = (1024, 32000, 32768, 50257, 65536, 100277, 128256, 151669, 152064, 200019, 256000)
LARGEST = 2.2e9          # bytes of logits


def draw(rng):
    kind = rng.choices([k for k, _ in KINDS], [w for _, w in KINDS])[0]
    dtype = rng.choice(("bf16", "bf16", "bf16", "f32"))
    esz = 4 if dtype == "f32" else 2
    V = rng.choice(VOCABULARIES) if rng.random() < 0.6 else int(math.exp(rng.uniform(math.log(1000), math.log(256001))))
    if kind == "loop":
        V = int(math.exp(rng.uniform(math.log(2000), math.log(20001))))          # (two tables of V rows)
    if kind not in ANY_V or rng.random() < 0.5:
        V = (V + 7) // 8 * 8
    gamma = rng.choice((1, 2, 3, 4, 5, 6, 8, 8, 10, 12, 16))
    rows = 1 if kind == "sample" else 2 * gamma + 1
    # (the cost of a row with no 16-byte vectors is not bound by its bytes, and host logits cross a slower link)
    most = LARGEST if V * esz % 16 == 0 else LARGEST / 8
    if kind in VERIFY_HOST:
        most = 6e7
    if kind == "loop":
        most = 3e8
    top = max(1, min(2048 if kind == "sample" else 512, int(most / (rows * V * esz))))
    B = int(math.exp(rng.uniform(0.0, math.log(top + 0.99))))
    head = rng.choice(("zipf", "zipf", "broad", "boost"))
    c = _case(None, kind, B, gamma, V, dtype=dtype, temperature=rng.choice((0.6, 0.8, 1.0, 1.0, 1.3)),
              sigma_d=rng.choice((0.1, 0.3, 0.7, 1.0, 1.5, 3.0)), head=head,
              masked=kind not in VERIFY_PROBS and rng.random() < 0.2, iters=rng.choice((4, 6, 8)) if kind == "loop" else 0)
    return c


def _rows(gen, shape, head):
    """Target logits in fp32: a Zipf law over randomly placed ranks with a little noise ("zipf"), the same under
    strong noise ("broad"), or Gaussian logits with about 50 strong tokens a row ("boost")."""
    V = shape[-1]
    if head == "boost":
        t = torch.randn(shape, generator=gen, device="cuda") * 3.0
        hot = torch.randint(0, V, (*shape[:-1], min(50, V)), generator=gen, device="cuda")
        return t.scatter_add_(-1, hot, torch.full(hot.shape, 8.0, device="cuda"))
    t = torch.randn(shape, generator=gen, device="cuda") * (0.3 if head == "zipf" else 3.0)
    rank = (1.0 - torch.rand(shape, generator=gen, device="cuda")) * V
    return t.sub_(rank.clamp_(min=1.0).log_().mul_(1.1))


def _mask(z):
    """Keeps about the largest tenth of every row (the tokens above a tenth's quantile of a sample of the row)."""
    V = z.shape[-1]
    seen = z[..., :: max(1, V // 1024)].sort(dim=-1).values
    cut = seen[..., int(0.9 * (seen.shape[-1] - 1))].unsqueeze(-1)
    return z.masked_fill_(z < cut, float("-inf"))


def _pick(gen, z, temperature):
    """One token per row from softmax(z / temperature) (the largest of z / T plus Gumbel noise)."""
    noise = (1.0 - torch.rand(z.shape, generator=gen, device="cuda")).log_().neg_().clamp_(min=1e-20).log_()
    return (z / temperature - noise).argmax(dim=-1).to(torch.int32)


def _tables(case, gen):
    V, td = case["V"], torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    tgt = torch.empty((V, V), dtype=td, device="cuda")
    drf = torch.empty((V, V), dtype=td, device="cuda")
    step = max(1, (1 << 26) // V)
    for r in range(0, V, step):
        t = _rows(gen, (min(step, V - r), V), case["head"])
        d = t + torch.randn(t.shape, generator=gen, device="cuda") * case["sigma_d"]
        if case["masked"]:
            t, d = _mask(t), _mask(d)
        tgt[r:r + step], drf[r:r + step] = t, d
    return tgt, drf


def prepare(case, seed):
    kind, B, g, V, T = case["kind"], case["B"], case["gamma"], case["V"], case["temperature"]
    td = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    uniform = lambda *shape: torch.rand(shape, generator=gen, device="cuda")
    state = dict(kind=kind, gamma=g, temperature=T)
    if kind == "loop":
        state["target"], state["draft"] = _tables(case, gen)
        state["first"] = torch.randint(0, V, (B,), generator=gen, device="cuda").to(torch.int32)
        state["u_draft"], state["u_verify"] = uniform(case["iters"], g, B), uniform(case["iters"], B, g + 2)
        return state
    if kind == "sample":
        state["logits"] = torch.empty((B, V), dtype=td, device="cuda")
        step = max(1, (1 << 26) // V)
        for b in range(0, B, step):
            z = _rows(gen, (min(step, B - b), V), case["head"])
            z.add_(torch.randn(z.shape, generator=gen, device="cuda"), alpha=case["sigma_d"])
            state["logits"][b:b + step] = _mask(z) if case["masked"] else z
        state["uniforms"] = uniform(B)
        return state
    tgt = torch.empty((B, g + 1, V), dtype=td, device="cuda")
    drf = torch.empty((B, g, V), dtype=td, device="cuda")
    tok = torch.empty((B, g), dtype=torch.int32, device="cuda")
    lse = torch.empty((B, g), dtype=torch.float32, device="cuda")
    step = max(1, (1 << 26) // ((g + 1) * V))
    for b in range(0, B, step):
        t = _rows(gen, (min(step, B - b), g + 1, V), case["head"])
        d = t[:, :g] + torch.randn((t.shape[0], g, V), generator=gen, device="cuda") * case["sigma_d"]
        if case["masked"]:
            t, d = _mask(t), _mask(d)
        tgt[b:b + step], drf[b:b + step] = t, d
        z = drf[b:b + step].float()                       # (the tokens are drawn from the logits as stored)
        tok[b:b + step] = _pick(gen, z, T)
        if kind in VERIFY_LSE:
            lse[b:b + step] = torch.logsumexp(z / T, dim=-1)
        if kind in VERIFY_PROBS:
            tgt[b:b + step] = torch.softmax(tgt[b:b + step].float() / T, dim=-1)
            drf[b:b + step] = torch.softmax(z / T, dim=-1)
    state.update(target=tgt, draft=drf, tokens=tok, uniforms=uniform(B, g + 2))
    if kind in VERIFY_LSE:
        state["lse"] = lse
    if kind in VERIFY_HOST:
        for k in ("target", "draft", "tokens", "uniforms"):
            state[k] = state[k].cpu().pin_memory()
        state["out_tokens"] = torch.empty((B, g + 1), dtype=torch.int32).pin_memory()
        state["out_len"] = torch.empty((B,), dtype=torch.int32).pin_memory()
    return state


def run(s):
    kind, T = s["kind"], s["temperature"]
    if kind == "loop":
        return specdec.run(s["target"], s["draft"], s["first"], s["u_draft"], s["u_verify"], s["gamma"], T)
    if kind == "sample":
        return bv.bv_sample_draft(s["logits"], s["uniforms"], T)
    if kind in VERIFY_HOST:
        return VERIFY_HOST[kind](s["target"], s["draft"], s["tokens"], s["uniforms"], T, s["out_tokens"], s["out_len"])
    if kind in VERIFY_LSE:
        return VERIFY_LSE[kind](s["target"], s["draft"], s["tokens"], s["uniforms"], s["lse"], T)
    if kind in VERIFY_PROBS:
        return VERIFY_PROBS[kind](s["target"], s["draft"], s["tokens"], s["uniforms"])
    return VERIFY[kind](s["target"], s["draft"], s["tokens"], s["uniforms"], T)


def work(case):
    """Rows that must be read once whatever the outcome: both models' rows and the last target row (Algorithms 2 and
    4), the target rows and one draft row (supplied normalisers), one row pair a sequence (Algorithm 1, which may stop
    at once, and probabilities, of which only the selected position is swept); about four operations a logit."""
    kind, B, g, V = case["kind"], case["B"], case["gamma"], case["V"]
    if kind == "loop":
        n = case["iters"] * B * (2 * g + 1)
        small = case["iters"] * B * (g + 2) * 12
    elif kind == "sample":
        n, small = B, 12 * B
    else:
        rows = {"block_lse": g + 2, "token_lse": 2, "token": 2, "block_probs": 2, "token_probs": 2, "token_host": 2}
        n, small = B * rows.get(kind, 2 * g + 1), B * (3 * g + 4) * 4
    return {"bytes": float(n * V * (4 if case["dtype"] == "f32" else 2) + small), "flops": 4.0 * n * V}


def exact(case, seed):
    """The normalisers of the drafting step and the intermediates of "block_ex" (p_i, S_i, h_i, log-normalisers) in
    64 bits, from the inputs as stored; tokens and lengths have no such value."""
    kind, T = case["kind"], case["temperature"]
    if kind not in ("sample", "block_ex"):
        return None
    s = prepare(case, seed)
    if kind == "sample":
        z = s["logits"]
        return None, torch.cat([torch.logsumexp(z[b:b + 16].double() / T, dim=-1) for b in range(0, z.shape[0], 16)])
    B, g = s["tokens"].shape
    f = lambda *shape: torch.empty(shape, dtype=torch.float64, device="cuda")
    p, S, h, lse_t, lse_d = f(B, g + 1), f(B, g), f(B, g + 1), f(B, g + 1), f(B, g)
    for b in range(B):
        P, Q = (torch.log_softmax(s[k][b].double() / T, dim=-1) for k in ("target", "draft"))
        lse_t[b] = torch.logsumexp(s["target"][b].double() / T, dim=-1)
        lse_d[b] = torch.logsumexp(s["draft"][b].double() / T, dim=-1)
        x = s["tokens"][b].long().unsqueeze(1)
        ratio = (P[:g].gather(1, x) - Q.gather(1, x)).exp().squeeze(1)
        p[b, 0] = 1.0
        for i in range(g):
            p[b, i + 1] = (p[b, i] * ratio[i]).clamp(max=1.0)
        S[b] = (p[b, :g, None] * P[:g].exp() - Q.exp()).clamp_(min=0.0).sum(dim=-1)
    h[:, :g] = torch.where(S > 0.0, S / (S + 1.0 - p[:, :g]), torch.zeros_like(S))
    h[:, 0], h[:, g] = 1.0, p[:, g]
    return None, None, dict(p=p, S=S, h=h, lse_t=lse_t, lse_d=lse_d)


def tolerance(case):
    """Whole values: sums in another order move the edges of the sampler's cells, and a uniform that close to one of
    the V edges picks the neighbour.  1e-4 + 2e-8 V of the draws is the bound that the library's tests use (seen
    against sums in 64 bits: 2 of 4096 draws at V = 128256, 1 of 4096 at 32000); a small batch has one to lose, and in
    the loop a sequence's later tokens follow the one that changed.
    Floating values, seen against 64 bits: 1.5e-7 for the normalisers, 1.2e-6 (1.4e-5 the worst single value) for the
    acceptance weights and residual masses of a close draft, which are differences of nearly equal sums of 32-bit terms."""
    values = case["B"] * (1 if case["kind"] == "sample" else case["gamma"] + 1)
    differ = 0.0099 if case["kind"] == "loop" else min(0.0099, max(1e-4 + 2e-8 * case["V"], 1.5 / values))
    if case["kind"] == "block_ex":
        return {"rel": 5e-6, "max": 6e-5, "differ": differ}
    return {"rel": 6e-7, "max": 1e-6, "differ": differ}
