"""The work that users of the library have it do, as timed cases over its public entry points.

Five kinds of pass:
  round   one draft-verify-accept round (`Session.sdd_step`) of a request being served; a finished request is followed
          by the next one in the same session (`Session.sdd_reset`), as a server does
  ar      one token of plain autoregressive decoding (`Session.sdd_ar_step`), requests following one another likewise
  sps     one round of the speculative-decoding warm start (`Session.sdd_sps_step`), likewise
  first   a new request up to its first token: `Session.sdd_reset` (prompt upload, prefill) and one `sdd_ar_step`
  accept  the acceptance step on a caller's own logits (`sdd_accept_logits`, `sdd_accept_logits_static`)

The networks are random-init (matrices N(0, 0.02^2)), the prompts uniform ids, the acceptance step's logits Gaussian with
a component that both models share; everything comes from the seed.
"""
from __future__ import annotations

import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2408_05636_b200 as sdd

PER_LAYER = ("ln1_g", "ln1_b", "w_qkv", "b_qkv", "w_o", "b_o", "ln2_g", "ln2_b", "w_fc1", "b_fc1", "w_fc2", "b_fc2")

# pairs of networks: target layers / heads / head width, drafter layers / heads / head width
_TINY = dict(lp=2, hp=4, dhp=64, lq=2, hq=4, dhq=32, V=512)
_SMALL = dict(lp=12, hp=12, dhp=64, lq=12, hq=12, dhq=64, V=50257)        # GPT-2 small and a drafter of its size
_XL = dict(lp=48, hp=25, dhp=64, lq=24, hq=16, dhq=64, V=50257)           # GPT-2 XL and a 300M drafter


def _pair(kind, name, net, dtype, prompt, gamma, T, batch, tau, max_new, ragged=False):
    return dict(net, name=name, kind=kind, dtype=dtype, prompt=prompt, gamma=gamma, T=T, batch=batch, tau=tau,
                max_new=max_new, ragged=ragged)


def listed():
    return [
        # one conversation's acceptance step between a user's own two models: launch latency and the call itself
        dict(name="accept_1x5", kind="accept", rows=1, gamma=5, V=50257, tau=1.0, static=False),
        # greedy acceptance of a few conversations in a host that may not allocate, vocabulary of another tokenizer
        dict(name="accept_7x15_greedy", kind="accept", rows=7, gamma=15, V=32003, tau=0.0, static=True),
        # a serving batch: streams 836 MB of logits
        dict(name="accept_64x32", kind="accept", rows=64, gamma=32, V=50257, tau=1.0, static=False),
        # the smallest networks, fp32: a round is a chain of tiny launches
        _pair("round", "round_tiny_fp32", _TINY, "fp32", 32, 8, 4, 1, 1.0, 64),
        # the paper's own setting: fp32, greedy, two denoising steps, gamma 15, one conversation
        _pair("round", "round_small_fp32", _SMALL, "fp32", 300, 15, 2, 1, 0.0, 64),
        # one conversation on the small pair
        _pair("round", "round_small_bf16", _SMALL, "bf16", 256, 16, 8, 1, 1.0, 64),
        # six conversations of different lengths, few denoising steps
        _pair("round", "round_small_b6_ragged", _SMALL, "bf16", 701, 20, 2, 6, 0.7, 64, ragged=True),
        # one conversation on the large pair
        _pair("round", "round_xl", _XL, "bf16", 512, 32, 16, 1, 1.0, 64),
        # a serving batch on the large pair: the largest case
        _pair("round", "round_xl_b16", _XL, "bf16", 1024, 16, 8, 16, 1.0, 64),
        # plain decoding of the large target, the loop that drafting competes with
        _pair("ar", "ar_xl", _XL, "bf16", 512, 16, 1, 1, 1.0, 64),
        # the start of a generation: five sequential evaluations of an autoregressive drafter, then verification
        _pair("sps", "sps_xl", _XL, "bf16", 100, 5, 1, 1, 1.0, 64),
        # time to the first token of four new requests of different lengths
        _pair("first", "first_xl_b4", _XL, "bf16", 1000, 16, 1, 4, 1.0, 16, ragged=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("accept", "accept", "round", "round", "round", "round", "ar", "sps", "first"))
    if kind == "accept":
        rows, gamma, V = _log_int(rng, 1, 64), _log_int(rng, 1, 128), _log_int(rng, 500, 152064)
        rows = max(1, min(rows, int(836e6 / 4 / ((2 * gamma + 1) * V))))
        # the library's own scratch holds 2 MiB of statistics
        static = rng.random() < 0.3 and rows * (2 * gamma + 1) * ((V + 3 + 8191) // 8192) * 8 <= sdd.ACCEPT_STATIC_SCRATCH_BYTES
        return dict(kind=kind, rows=rows, gamma=gamma, V=V, tau=rng.choice((0.0, 0.7, 1.0, 1.0)), static=static)
    fp32 = kind == "round" and rng.random() < 0.35
    c = dict(
        kind=kind, dtype="fp32" if fp32 else "bf16",
        lp=_log_int(rng, 2, 12 if fp32 else 48), hp=_log_int(rng, 2, 12 if fp32 else 25), dhp=64,
        lq=_log_int(rng, 2, 12 if fp32 else 24), hq=_log_int(rng, 2, 12 if fp32 else 16), dhq=rng.choice((32, 64)) if fp32 else 64,
        V=_log_int(rng, 500, 50300), prompt=_log_int(rng, 16, 1024), gamma=_log_int(rng, 1, 8 if kind == "sps" else 64),
        T=_log_int(rng, 1, 16) if kind == "round" else 1, batch=_log_int(rng, 1, 4 if fp32 else 16),
        tau=rng.choice((0.0, 0.7, 1.0, 1.0)), max_new=_log_int(rng, 16, 128), ragged=rng.random() < 0.5)
    if kind == "sps":
        c["hq"] = min(c["hq"], c["hp"])            # the warm start's drafter is no wider than the target
    limit = 6e11 if fp32 else 6e13
    while work(c)["flops"] > limit:                # no case costs more than the largest listed one
        if c["batch"] > 1:
            c["batch"] -= 1
        elif c["prompt"] > 64:
            c["prompt"] = c["prompt"] * 3 // 4
        else:
            c["T"] = max(1, c["T"] - 1)
    return c


# ---- inputs -----------------------------------------------------------------------------------------------------------
class _Weights:
    """A random-init network whose tensors were made on the GPU, in the library's tensor order."""

    def __init__(self, gen, vocab, n_layer, d, n_head, n_ctx, causal, dtype):
        wide = torch.bfloat16 if dtype == "bf16" else torch.float32

        def normal(*shape, std=0.02, mean=0.0, to=torch.float32):
            return (torch.randn(*shape, device="cuda", generator=gen) * std + mean).to(to)

        shapes = {"w_qkv": (3 * d, d), "w_o": (d, d), "w_fc1": (4 * d, d), "w_fc2": (d, 4 * d),
                  "b_qkv": (3 * d,), "b_o": (d,), "b_fc1": (4 * d,), "b_fc2": (d,)}
        self.keep = [normal(vocab + (0 if causal else 1), d, to=wide), normal(n_ctx, d, to=wide)]
        for _ in range(n_layer):
            for n in PER_LAYER:
                if n.startswith("ln"):
                    self.keep.append(normal(d, mean=1.0 if n.endswith("_g") else 0.0))
                else:
                    self.keep.append(normal(*shapes[n], to=wide if n.startswith("w_") else torch.float32))
        self.keep += [normal(d, mean=1.0), normal(d)]
        self.shape = SimpleNamespace(vocab=vocab, n_layer=n_layer, d_model=d, n_head=n_head, n_ctx=n_ctx, causal=causal)
        self.ptrs = (ctypes.c_void_p * len(self.keep))(*[t.data_ptr() for t in self.keep])
        self.c = sdd.sdd_model(vocab, n_layer, d, n_head, n_ctx, 1 if causal else 0,
                               sdd.SDD_BF16 if dtype == "bf16" else sdd.SDD_FP32,
                               ctypes.cast(self.ptrs, ctypes.POINTER(ctypes.c_void_p)), len(self.keep))


def _prepare_accept(case, gen):
    rows, gamma, V = case["rows"], case["gamma"], case["V"]
    lp = torch.randn(rows, gamma + 1, V, device="cuda", generator=gen)
    lq = lp[:, :gamma] + 0.5 * torch.randn(rows, gamma, V, device="cuda", generator=gen)
    lp += 0.5 * torch.randn(rows, gamma + 1, V, device="cuda", generator=gen)
    ids = torch.empty(rows, gamma, dtype=torch.int32, device="cuda")
    for r in range(rows):                          # the drafts are draws from the drafter's own distribution
        z = lq[r] if case["tau"] == 0 else lq[r] / case["tau"] - torch.log(-torch.log(
            torch.rand(gamma, V, device="cuda", generator=gen).clamp_(1e-7, 1 - 1e-7)))
        ids[r] = z.argmax(-1)
    s = SimpleNamespace(kind="accept", lp=lp, lq=lq, ids=ids, tau=case["tau"], static=case["static"], round=0,
                        seed=int(torch.randint(0, 1 << 30, (1,), device="cuda", generator=gen).item()))
    if s.static:
        s.n = torch.empty(rows, dtype=torch.int32, device="cuda")
        s.out = torch.empty(rows, gamma + 1, dtype=torch.int32, device="cuda")
        s.prob = torch.empty(rows, gamma, device="cuda")
    return s


_streams = []


def _stream():
    """The one stream of the program: its sessions' rounds follow one another."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "accept":
        s = _prepare_accept(case, gen)
        torch.cuda.synchronize()
        return s
    rng = np.random.default_rng(seed)
    B, V, gamma, dtype = case["batch"], case["V"], case["gamma"], case["dtype"]
    longest = case["prompt"] + case["max_new"] + gamma
    n_ctx = 128 if longest <= 128 else 1024 if longest <= 1024 else 2048
    target = _Weights(gen, V, case["lp"], case["hp"] * case["dhp"], case["hp"], n_ctx, True, dtype)
    drafter = _Weights(gen, V, case["lq"], case["hq"] * case["dhq"], case["hq"], n_ctx, False, dtype)
    plen = [case["prompt"]] * B
    if case["ragged"]:
        plen = [case["prompt"]] + [int(n) for n in rng.integers(max(2, case["prompt"] // 4), case["prompt"] + 1, B - 1)]
    s = SimpleNamespace(kind=case["kind"], gamma=gamma, max_new=case["max_new"], plen=plen,
                        prompts=rng.integers(0, V, (B, case["prompt"]), dtype=np.int32))
    torch.cuda.synchronize()
    s.sess = sdd.Session(target, drafter, s.prompts, plen, gamma, case["T"], case["max_new"], case["tau"], case["tau"], seed,
                         stream=_stream())
    if case["kind"] == "sps":
        s.sess.sdd_sps_attach(_Weights(gen, V, case["lq"], case["hq"] * case["dhq"], case["hq"], n_ctx, True, dtype))
    rows_p = 1 if case["kind"] in ("ar", "first") else gamma + 1
    s.outputs = {
        "tokens": s.sess.sdd_tap(sdd.TAP_TOKENS),
        # the target's scores of the token after the context, and the drafter's of the draft (its first token only in the
        # warm start, where each further one depends on the tokens drawn before it)
        "p": s.sess.sdd_tap(sdd.TAP_LOGITS_P)[: B * rows_p * V].view(B, rows_p, V)[:, 0],
    }
    if case["kind"] in ("round", "sps"):
        q = s.sess.sdd_tap(sdd.TAP_Q_LOGITS).view(B, gamma, V)
        s.outputs["q"] = q if case["kind"] == "round" else q[:, 0]
    torch.cuda.synchronize()
    return s


# ---- one pass ---------------------------------------------------------------------------------------------------------
def run(s):
    if s.kind == "accept":
        s.round += 1
        if s.static:
            sdd.sdd_accept_logits_static(s.lp, s.lq, s.ids, s.n, s.out, s.prob, s.tau, s.tau, s.seed, s.round)
            return s.n, s.out, s.prob
        return sdd.sdd_accept_logits(s.lp, s.lq, s.ids, s.tau, s.tau, s.seed, s.round)
    sess = s.sess
    if s.kind == "first":
        sess.sdd_reset(s.prompts, s.plen)
        sess.sdd_ar_step()
        return s.outputs
    if sess.sdd_progress()[1] >= s.max_new:        # every sequence of the batch has its tokens: the next requests
        sess.sdd_reset(s.prompts, s.plen)
    if s.kind == "round":
        sess.sdd_step()
    elif s.kind == "ar":
        sess.sdd_ar_step()
    else:
        sess.sdd_sps_step(s.gamma)
    return s.outputs


# ---- what a pass cannot do without ---------------------------------------------------------------------------------------
def work(case):
    if case["kind"] == "accept":
        rows, gamma, V = case["rows"], case["gamma"], case["V"]
        per_row = (gamma + 1 if case["tau"] == 0 else 2 * gamma + 1) * V    # greedy acceptance needs the target's rows only
        return {"bytes": rows * (4.0 * per_row + 4.0 * (3 * gamma + 2)), "flops": 2.0 * rows * per_row}
    B, V, gamma, T = case["batch"], case["V"], case["gamma"], case["T"]
    e = 2 if case["dtype"] == "bf16" else 4
    dp, dq, lp, lq = case["hp"] * case["dhp"], case["hq"] * case["dhq"], case["lp"], case["lq"]
    c = case["prompt"] * (1.0 if not case["ragged"] else (1 + 0.625 * (B - 1)) / B)       # mean context length
    body_p, body_q = 12.0 * dp * dp * lp, 12.0 * dq * dq * lq                             # parameters of the blocks

    def target(rows, keys, head_rows):
        """`rows` new tokens per sequence against `keys` keys in all."""
        flops = 2 * B * rows * body_p + 4 * B * rows * keys * dp * lp + 2 * B * head_rows * V * dp
        nbytes = body_p * e + (V * dp * e if head_rows else 0) + 2 * B * keys * dp * lp * e + 4 * B * head_rows * V
        return flops, nbytes

    if case["kind"] == "first":
        f1, b1 = target(c - 1, c / 2, 0)
        f2, b2 = target(1, c, 1)
        return {"flops": f1 + f2, "bytes": b1 + b2}
    if case["kind"] == "ar":
        f, b = target(1, c, 1)
        return {"flops": f, "bytes": b}
    f, b = target(gamma + 1, c + gamma, gamma + 1)
    if case["kind"] == "sps":
        # the drafter's weights are read again for every evaluation: each depends on the token drawn from the one before
        fq = 2 * B * body_q + 4 * B * c * dq * lq + 2 * B * V * dq
        bq = body_q * e + V * dq * e + 2 * B * c * dq * lq * e + 4 * B * V
        return {"flops": f + gamma * fq, "bytes": b + gamma * bq}
    # evaluations of a round whose input differs from the one before: every slot is revealed at a step uniform on 1..T
    evals = 1 + (T - 1) * (1 - (1 - 1 / T) ** (B * gamma)) if T > 1 else 1
    L = c + gamma
    fq = 2 * B * L * body_q + 4 * B * L * L * dq * lq + 2 * B * gamma * V * dq
    bq = body_q * e + V * dq * e + 4 * B * gamma * V
    return {"flops": f + evals * fq, "bytes": b + evals * bq}


def tolerance(case):
    if case["kind"] == "accept":
        # fp32 probabilities out of fp32 log-sum-exps; a draw whose two best scores agree to fp32 may fall either way
        return {"rel": 1e-5, "differ": 0.02}
    # Scores in the networks' own precision.  A draw or a test within rounding of a tie moves one token and what follows
    # it in that sequence's round: allowed for one sequence, and one in eight of a larger batch.
    stride = case["prompt"] + case["max_new"] + case["gamma"]
    stride = 128 if stride <= 128 else 1024 if stride <= 1024 else 2048
    emitted = 1 if case["kind"] in ("ar", "first") else case["gamma"] + 1
    B = case["batch"]
    return {"rel": 1e-2 if case["dtype"] == "bf16" else 1e-5, "differ": -(-B // 8) * emitted / (B * stride)}
