"""The work that a user of this library has it do, as cases that can be timed.

Four kinds, all through the public entry points of paper_2402_11809_b200.binding, with the argument
structs and buffers kept from call to call as a decoding program keeps them:

  step    one auto-correct decoding step on the GPU: space_attn_step, then space_verify_commit
          (greedy, sampling, or sampling with top-k / top-p; contiguous or paged cache)
  lmhead  the end of the model call from hidden states: space_lmhead_verify
  host    one step from host buffers: space_step_host with the cache resident on the device
  loop    several steps of the decoding loop with its state on the GPU, one after another:
          space_decode_begin, then space_attn_step, space_verify_commit, space_decode_advance per step
"""
import math

import numpy as np
import torch

from paper_2402_11809_b200 import binding as S

# logits of a planted candidate (the workloads of this repository use the same two values)
PLANT = {"greedy": 30.0, "sample": 16.0}
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}

MAX_KV_BYTES = 2.3e9          # the largest listed step reads about this much cache
MAX_ATTN_FLOPS = 1.0e11
MAX_LOGIT_BYTES = 4.2e8
MAX_LMHEAD_FLOPS = 6.0e11


def _step(name, B, heads, d, L, k, V, logits="bf16", out="bf16", mode="greedy", temperature=1.0,
          accept=(0.8, 0.8), top_k=0, top_p=1.0, resample=0, paged=False):
    return dict(name=name, kind="step", B=B, H_q=heads[0], H_kv=heads[1], d=d, L_lo=L[0], L_hi=L[1], k=k, V=V,
                logits=logits, out=out, mode=mode, temperature=temperature, p_lo=accept[0], p_hi=accept[1],
                top_k=top_k, top_p=top_p, resample=resample, paged=paged)


def _lmhead(name, B, k, V, D, mode="greedy", temperature=1.0, resample=0, accept=0.8):
    return dict(name=name, kind="lmhead", B=B, k=k, V=V, D=D, mode=mode, temperature=temperature,
                resample=resample, p_lo=accept, p_hi=accept)


def listed():
    return [
        # the smallest step: a short chat turn on a small model, where launches and latency are all there is
        _step("tiny", 1, (8, 8), 64, (128, 128), 4, 1000, logits="f32", out="f32", accept=(0.7, 0.7)),
        # the headline workload: one user of a 7B-shaped model, 2k tokens in, one layer's attention and the verify
        _step("llama7b", 1, (32, 32), 128, (2048, 2048), 5, 32000),
        # a server's batch of users at ragged lengths, fp32 attention output
        _step("ragged16", 16, (32, 32), 128, (512, 4096), 5, 32000, out="f32", accept=(0.3, 0.9)),
        # a 70B-shaped model with grouped queries at long context: the contraction is large
        _step("gqa70b", 8, (64, 8), 128, (8192, 8192), 6, 32000),
        # the largest step: 64 users, lengths up to 16k, large vocabulary, rejection sampling
        _step("sampling64", 64, (32, 8), 128, (1024, 16384), 4, 128256, mode="sample", temperature=0.8),
        # continuous batching on a paged cache, short drafts, top-k 10 / top-p 0.95 with compact draft lists
        _step("paged_top10", 24, (32, 8), 128, (200, 6000), 2, 128256, mode="sample", temperature=0.8,
              top_k=10, top_p=0.95, resample=2, paged=True),
        # odd sizes throughout: a vocabulary whose rows are not 16-byte aligned, short ragged lengths, head size 64
        _step("odd5", 5, (16, 8), 64, (37, 1999), 3, 50257, accept=(0.3, 0.9)),
        # output projection and verification from hidden states, one user of a 7B-shaped model
        _lmhead("lmhead_llama7b", 1, 5, 32000, 4096),
        # the same for a small batch (144 block rows)
        _lmhead("lmhead_batch4", 4, 5, 32000, 4096),
        # the largest projection: 16 users, large vocabulary, sampling
        _lmhead("lmhead_batch16", 16, 5, 128256, 4096, mode="sample", temperature=0.8),
        # a program that holds q, logits and new cache rows in host memory: copies in, the step, copies out
        dict(name="host_resident", kind="host", B=1, H_q=32, H_kv=32, d=128, L_lo=2048, L_hi=2048, k=5, V=32000,
             logits="bf16", mode="greedy", p_lo=0.8, p_hi=0.8),
        # eight decoding steps one after another for two users of a 7B-shaped model
        dict(name="decode_loop", kind="loop", B=2, H_q=32, H_kv=32, d=128, L_lo=500, L_hi=1500, k=5, V=32000,
             steps=8, p_lo=0.8, p_hi=0.8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _heads(rng):
    H_kv = rng.choice([1, 2, 4, 8, 8, 16, 32])
    G = rng.choice([g for g in (1, 1, 2, 4, 8) if H_kv * g <= 64])
    return H_kv * G, H_kv


def _vocab(rng):
    return rng.choice([32000, 50257, 128256, _log_int(rng, 1000, 128256), _log_int(rng, 1000, 128256) | 1])


def draw(rng):
    kind = rng.choice(["greedy", "greedy", "greedy", "sample", "filtered", "lmhead", "lmhead", "host", "loop"])
    k = rng.randint(1, 7)
    n_q = (k + 1) * (k + 1)
    if kind == "lmhead":
        D = 8 * rng.randint(64, 640) if rng.random() < 0.3 else 64 * rng.randint(8, 80)
        V = min(_vocab(rng), int(1.05e9 / (2 * D)))
        most = max(1, min(16, int(MAX_LMHEAD_FLOPS / (2.0 * n_q * V * D))))
        sample = rng.random() < 0.4
        c = _lmhead("", _log_int(rng, 1, most), k, V, D, mode="sample" if sample else "greedy",
                    temperature=round(rng.uniform(0.6, 1.2), 2) if sample else 1.0,
                    resample=rng.choice([0, 1]) if sample else 0, accept=round(rng.uniform(0.3, 0.9), 2))
        del c["name"]
        return c
    H_q, H_kv = _heads(rng)
    d = rng.choice([64, 128, 128])
    hi = _log_int(rng, 64, 16384)
    lo = hi if rng.random() < 0.3 else max(1, int(hi * rng.uniform(0.05, 0.9)))
    V = _vocab(rng)
    p = sorted(round(rng.uniform(0.3, 0.9), 2) for _ in range(2))
    if kind in ("host", "loop"):
        hi, lo = min(hi, 4096), min(lo, 4096)
        k = min(k, 6)
        c = dict(kind=kind, B=_log_int(rng, 1, 4), H_q=H_q, H_kv=H_kv, d=d, L_lo=lo, L_hi=hi, k=k, V=V,
                 p_lo=p[0], p_hi=p[1])
        if kind == "host":
            c.update(logits=rng.choice(["bf16", "bf16", "f32"]), mode="greedy")
        else:
            c.update(steps=8)
        return c
    most = 64
    most = min(most, MAX_KV_BYTES / ((hi + n_q) * H_kv * d * 4.0), MAX_ATTN_FLOPS / (4.0 * n_q * H_q * (hi + n_q) * d),
               MAX_LOGIT_BYTES / (4.0 * n_q * V))
    B = _log_int(rng, 1, max(1, int(most)))
    c = _step("", B, (H_q, H_kv), d, (lo, hi), k, V, logits=rng.choice(["bf16", "bf16", "f32"]),
              out=rng.choice(["bf16", "f32"]), accept=(p[0], p[1]), paged=rng.random() < 0.35)
    if kind != "greedy":
        c.update(mode="sample", temperature=round(rng.uniform(0.6, 1.2), 2), resample=rng.choice([0, 0, 1]))
    if kind == "filtered":
        c.update(top_k=rng.randint(5, 32), top_p=round(rng.uniform(0.85, 1.0), 2), resample=rng.choice([0, 2, 2]))
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _generators(seed):
    return torch.Generator(device="cuda").manual_seed(seed), np.random.Generator(np.random.Philox(key=seed))


def _normal(g, shape, dtype, sigma=1.0):
    x = torch.randn(shape, dtype=dtype, device="cuda", generator=g)
    return x.mul_(sigma) if sigma != 1.0 else x


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _int(*shape):
    return torch.zeros(shape, dtype=torch.int32, device="cuda")


def _planted(rng, B, k, p_lo, p_hi):
    return rng.uniform(size=(B, k)) < rng.uniform(p_lo, p_hi, size=B)[:, None]


def _lengths(rng, c):
    return rng.integers(c["L_lo"], c["L_hi"] + 1, size=c["B"]).astype(np.int32)


def _results(B, k):
    return dict(n_accept=_int(B), out_tokens=_int(B, k + 1), n_out=_int(B), next_cand=_int(B, k),
                next_cand_prob=torch.zeros(B, k, device="cuda"),
                finished=torch.zeros(B, dtype=torch.uint8, device="cuda"))


def _cache(g, rng, c, extra_rows):
    """K and V for lengths up to L_hi + extra_rows: contiguous, or pools behind a shuffled page table."""
    B, H, d = c["B"], c["H_kv"], c["d"]
    rows = c["L_hi"] + extra_rows
    if c.get("paged"):
        per_seq = -(-rows // S.PAGE_SIZE)
        n_pages = B * per_seq + 3
        table = _dev(rng.permutation(n_pages)[: B * per_seq].reshape(B, per_seq).astype(np.int32))
        shape, cap = (n_pages, H, S.PAGE_SIZE, d), per_seq * S.PAGE_SIZE
    else:
        cap = -(-rows // 64) * 64
        table, shape = None, (B, H, cap, d)
    return _normal(g, shape, torch.bfloat16), _normal(g, shape, torch.bfloat16), table, cap


def _prepare_step(c, seed):
    g, rng = _generators(seed)
    B, k, V, n_q = c["B"], c["k"], c["V"], (c["k"] + 1) ** 2
    kc, vc, table, cap = _cache(g, rng, c, n_q)
    ctx = S.Context(max_batch=B, n_q_heads=c["H_q"], n_kv_heads=c["H_kv"], head_dim=c["d"], k_max=k, vocab=V, s_cap=cap)
    q = _normal(g, (B, n_q, c["H_q"], c["d"]), torch.bfloat16)
    kv_len = _dev(_lengths(rng, c))
    logits = _normal(g, (B, n_q, V), DTYPES[c["logits"]], 3.0)
    cand = rng.integers(0, V, size=(B, k)).astype(np.int32)
    cand_prob = np.ones((B, k), dtype=np.float32)
    planted = _planted(rng, B, k, c["p_lo"], c["p_hi"])
    drafts = {}
    if c["resample"] == 2:
        # the lists that the step before handed on: descending probabilities, the candidate one of their
        # tokens; the target rows agree with them in part
        n = c["top_k"]
        tok = rng.integers(0, V, size=(B, k, n)).astype(np.int32)
        w = -np.sort(-rng.exponential(size=(B, k, n)) ** 2)
        prob = (w / w.sum(-1, keepdims=True)).astype(np.float32)
        pick = np.minimum((np.cumsum(prob, -1) < rng.uniform(size=(B, k, 1))).sum(-1), n - 1)
        cand = np.take_along_axis(tok, pick[..., None], -1)[..., 0].copy()
        cand_prob = np.take_along_axis(prob, pick[..., None], -1)[..., 0].copy()
        z = PLANT["sample"] + c["temperature"] * np.log(np.maximum(prob, 1e-6)) + 0.3 * rng.standard_normal(prob.shape)
        bb, ii = np.nonzero(planted)
        logits[_dev(np.repeat(bb, n)), _dev(np.repeat(ii * (k + 1), n)), _dev(tok[bb, ii].reshape(-1).astype(np.int64))] = \
            _dev(z[bb, ii].reshape(-1).astype(np.float32)).to(logits.dtype)
        drafts = dict(draft_tok=_dev(tok), draft_prob=_dev(prob), next_draft_tok=_int(B, k, n),
                      next_draft_prob=torch.zeros(B, k, n, device="cuda"))
    else:
        bb, ii = np.nonzero(planted)
        logits[_dev(bb), _dev(ii * (k + 1)), _dev(cand[bb, ii].astype(np.int64))] = PLANT[c["mode"]]
        if c["resample"] == 1:
            cand_prob = rng.uniform(0.3, 1.0, size=(B, k)).astype(np.float32)
    cand, cand_prob, seq_id = _dev(cand), _dev(cand_prob), _dev(np.arange(B, dtype=np.int32))
    out = torch.zeros(B, n_q, c["H_q"], c["d"], dtype=DTYPES[c["out"]], device="cuda")
    status, kv_new, r = _int(B), _int(B), _results(B, k)
    attn = ctx.attn_args(q, kc, vc, kv_len, out, k, 1.0 / math.sqrt(c["d"]), status=status, page_table=table)
    verify = ctx.verify_args(logits, cand, cand_prob, kv_len, k=k, seed=1234,
                             mode=S.MODE_SAMPLE if c["mode"] == "sample" else S.MODE_GREEDY,
                             temperature=c["temperature"], resample=c["resample"], seq_id=seq_id, status=status,
                             top_k=c["top_k"], top_p=c["top_p"], eos_id=2, **r, **drafts)
    commit = ctx.commit_args(kc, vc, r["n_accept"], kv_len, k, kv_len_out=kv_new, status=status, page_table=table)
    outputs = dict(r, out=out, k_cache=kc, v_cache=vc, kv_len=kv_new, status=status)
    outputs.update({n: t for n, t in drafts.items() if n.startswith("next")})
    return dict(kind="step", ctx=ctx, attn=attn, verify=verify, commit=commit, outputs=outputs,
                keep=(q, kv_len, logits, cand, cand_prob, seq_id, table, drafts))


def _prepare_lmhead(c, seed):
    g, rng = _generators(seed)
    B, k, V, D, n_q, k1 = c["B"], c["k"], c["V"], c["D"], (c["k"] + 1) ** 2, c["k"] + 1
    sigma = 3.0
    ctx = S.Context(max_batch=B, k_max=k, vocab=V, s_cap=4096)
    weight = _normal(g, (V, D), torch.bfloat16, sigma / math.sqrt(D))
    hidden = _normal(g, (B, n_q, D), torch.bfloat16)
    cand = rng.integers(0, V, size=(B, k)).astype(np.int32)
    bb, ii = np.nonzero(_planted(rng, B, k, c["p_lo"], c["p_hi"]))
    # a hidden row along the candidate's own embedding makes that token the row's likely one
    gain = PLANT[c["mode"]] / sigma ** 2
    at = (_dev(bb), _dev(ii * k1))
    hidden[at] = (gain * weight[_dev(cand[bb, ii].astype(np.int64))].float() + 0.05 * hidden[at].float()).bfloat16()
    cand_prob = np.ones((B, k), np.float32) if c["resample"] == 0 else rng.uniform(0.3, 1.0, size=(B, k)).astype(np.float32)
    cand, cand_prob = _dev(cand), _dev(cand_prob)
    seq_id, kv_len = _dev(np.arange(B, dtype=np.int32)), _dev(rng.integers(100, 4000, size=B).astype(np.int32))
    status, r = _int(B), _results(B, k)
    args = ctx.lmhead_args(hidden, weight, cand, k=k, eos_id=2, status=status, seed=1234, temperature=c["temperature"],
                           mode=S.MODE_SAMPLE if c["mode"] == "sample" else S.MODE_GREEDY, resample=c["resample"],
                           cand_prob=cand_prob, seq_id=seq_id, kv_len=kv_len, **r)
    return dict(kind="lmhead", ctx=ctx, args=args, outputs=dict(r, status=status),
                keep=(weight, hidden, cand, cand_prob, seq_id, kv_len))


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    return h.copy_(t)


def _prepare_host(c, seed):
    g, rng = _generators(seed)
    B, k, V, n_q = c["B"], c["k"], c["V"], (c["k"] + 1) ** 2
    kc, vc, _, cap = _cache(g, rng, c, n_q)
    ctx = S.Context(max_batch=B, n_q_heads=c["H_q"], n_kv_heads=c["H_kv"], head_dim=c["d"], k_max=k, vocab=V, s_cap=cap,
                    host_staging=1)
    logits = _normal(g, (B, n_q, V), DTYPES[c["logits"]], 3.0)
    cand = rng.integers(0, V, size=(B, k)).astype(np.int32)
    bb, ii = np.nonzero(_planted(rng, B, k, c["p_lo"], c["p_hi"]))
    logits[_dev(bb), _dev(ii * (k + 1)), _dev(cand[bb, ii].astype(np.int64))] = PLANT[c["mode"]]
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32)  # noqa: E731
    lengths = torch.from_numpy(_lengths(rng, c))
    h = dict(q=_pinned(_normal(g, (B, n_q, c["H_q"], c["d"]), torch.bfloat16)), k_cache=_pinned(kc), v_cache=_pinned(vc),
             logits=_pinned(logits), cand=torch.from_numpy(cand), cand_prob=torch.ones(B, k), kv_len=lengths.clone(),
             out=torch.zeros(B, n_q, c["H_q"], c["d"], pin_memory=True), n_accept=i32(B), out_tokens=i32(B, k + 1),
             n_out=i32(B), next_cand=i32(B, k), next_cand_prob=torch.zeros(B, k),
             finished=torch.zeros(B, dtype=torch.uint8), status=i32(B))
    args = S.HostStepArgs(batch=B, k=k, vocab=V, logits_dtype=S.DTYPE_F32 if c["logits"] == "f32" else S.DTYPE_BF16,
                          mode=S.MODE_GREEDY, resample=0, eos_id=2, mask_variant=S.MASK_SAME_GROUP,
                          scale=1.0 / math.sqrt(c["d"]), temperature=1.0, seed=1234, cache_resident=0, reserved=0,
                          **{n: t.data_ptr() for n, t in h.items()})
    ctx.space_step_host(args)          # the prefill's hand-over: the whole cache goes up once
    args.cache_resident = 1
    return dict(kind="host", ctx=ctx, args=args, kv_len=h["kv_len"], lengths=lengths, keep=h,
                outputs={n: h[n] for n in ("out", "k_cache", "v_cache", "kv_len", "n_accept", "out_tokens", "n_out",
                                           "next_cand", "next_cand_prob", "finished", "status")})


def _prepare_loop(c, seed):
    g, rng = _generators(seed)
    B, k, V, steps, n_q, k1 = c["B"], c["k"], c["V"], c["steps"], (c["k"] + 1) ** 2, c["k"] + 1
    kc, vc, _, cap = _cache(g, rng, c, n_q + steps * k1)
    ctx = S.Context(max_batch=B, n_q_heads=c["H_q"], n_kv_heads=c["H_kv"], head_dim=c["d"], k_max=k, vocab=V, s_cap=cap)
    kv_len0 = _dev(_lengths(rng, c))
    kv_len, kv_next, last = _int(B), _int(B), _dev(rng.integers(3, V, size=B).astype(np.int32))
    tokens, n_tokens, last_token = _int(B, steps * k1), _int(B), _int(B)
    cand, cand_prob = _int(B, k), torch.zeros(B, k, device="cuda")
    finished = torch.zeros(B, dtype=torch.uint8, device="cuda")
    block_tokens, block_pos = _int(B, n_q), _int(B, n_q)
    state = ctx.decode_state(tokens, n_tokens, last_token, cand, cand_prob, kv_len, finished, block_tokens, block_pos, k,
                             mask_token_id=V - 1)
    status, r = _int(B), _results(B, k)
    out = torch.zeros(steps, B, n_q, c["H_q"], c["d"], dtype=torch.bfloat16, device="cuda")
    q = _normal(g, (steps, B, n_q, c["H_q"], c["d"]), torch.bfloat16)
    logits = _normal(g, (steps, B, n_q, V), torch.bfloat16, 3.0)
    calls, follow = [], None
    for s in range(steps):
        # every group's mask rows propose the same next candidates; the next step's target rows agree with
        # each of them with the acceptance probability
        if follow is not None:
            bb, ii = np.nonzero(_planted(rng, B, k, c["p_lo"], c["p_hi"]))
            logits[s][_dev(bb), _dev(ii * k1), _dev(follow[bb, ii])] = PLANT["greedy"]
        follow = rng.integers(3, V, size=(B, k))
        for grp in range(k1):
            for o in range(k):
                logits[s][torch.arange(B, device="cuda"), grp * k1 + o + 1, _dev(follow[:, o])] = PLANT["greedy"]
        attn = ctx.attn_args(q[s], kc, vc, kv_len, out[s], k, 1.0 / math.sqrt(c["d"]), status=status)
        verify = ctx.verify_args(logits[s], cand, cand_prob, kv_len, k=k, eos_id=2, status=status, **r)
        commit = ctx.commit_args(kc, vc, r["n_accept"], kv_len, k, kv_len_out=kv_next, status=status)
        calls.append((attn, verify, commit))
    return dict(kind="loop", ctx=ctx, calls=calls, state=state, last=last, kv_len=kv_len, kv_len0=kv_len0,
                kv_next=kv_next, r=r, keep=(q, logits, last_token, cand, cand_prob),
                outputs=dict(tokens=tokens, n_tokens=n_tokens, kv_len=kv_len, finished=finished, out=out,
                             block_tokens=block_tokens, block_pos=block_pos, k_cache=kc, v_cache=vc, status=status))


def prepare(case, seed):
    return {"step": _prepare_step, "lmhead": _prepare_lmhead, "host": _prepare_host, "loop": _prepare_loop}[case["kind"]](case, seed)


# ---------------------------------------------------------------- one pass
def run(state):
    ctx, kind = state["ctx"], state["kind"]
    if kind == "step":
        ctx.space_attn_step(state["attn"])
        ctx.space_verify_commit(state["verify"], state["commit"])
    elif kind == "lmhead":
        ctx.space_lmhead_verify(state["args"])
    elif kind == "host":
        state["kv_len"].copy_(state["lengths"])          # the call moves the lengths on: the same step again
        ctx.space_step_host(state["args"])
    else:
        r = state["r"]
        state["kv_len"].copy_(state["kv_len0"])          # the prompt's length, as the prefill leaves it
        ctx.space_decode_begin(state["state"], state["last"])
        for attn, verify, commit in state["calls"]:
            ctx.space_attn_step(attn)
            ctx.space_verify_commit(verify, commit)
            ctx.space_decode_advance(state["state"], r["out_tokens"], r["n_out"], r["next_cand"], r["next_cand_prob"],
                                     r["finished"], state["kv_next"])
    return state["outputs"]


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    c = case
    B, k, V, n_q = c["B"], c["k"], c["V"], (c["k"] + 1) ** 2
    if c["kind"] == "lmhead":
        # the embedding once, every block row's hidden state once; the products of the 2k+1 rows that the
        # step decides on (target rows, then the mask rows of the selected group)
        return {"bytes": 2.0 * V * c["D"] + 2.0 * B * n_q * c["D"], "flops": 2.0 * B * (2 * k + 1) * V * c["D"]}
    keys = B * ((c["L_lo"] + c["L_hi"]) / 2.0 + n_q)
    esz = 4 if c.get("logits") == "f32" else 2
    osz = 4 if c["kind"] == "host" or c.get("out") == "f32" else 2
    kv = keys * c["H_kv"] * c["d"] * 4.0
    q_out = B * n_q * c["H_q"] * c["d"] * (2.0 + osz)
    rows = B * (2 * k + 1) * V * float(esz)
    moved = B * 0.5 * k * c["H_kv"] * c["d"] * 8.0         # accepted rows, read and written (about half of k)
    flops = 4.0 * n_q * c["H_q"] * keys * c["d"]
    n = c.get("steps", 1)                                  # a loop reads the cache once, the rest every step
    return {"bytes": kv + n * (q_out + rows + moved), "flops": n * flops}


def tolerance(case):
    if case["kind"] == "lmhead":
        # whole decisions, and probabilities from fp32 sums over the vocabulary
        return {"rel": 1e-4, "max": 4e-3, "differ": 5e-3 if case["mode"] == "sample" else 0.0}
    # attention over bf16 inputs with fp32 accumulation: an fp32 output carries the products' rounding, a bf16
    # output its own; whole decisions are equal except for ties of noisy scores in sampling
    f32 = case["kind"] == "host" or case.get("out") == "f32"
    return {"rel": 5e-4 if f32 else 4e-3, "max": 5e-3 if f32 else 3e-2,
            "differ": 5e-3 if case.get("mode") == "sample" else 0.0}
