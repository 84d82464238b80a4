"""GPU parity at the edges of the kernels' dispatch rules (row alignment, chunk and tile remainders, grouping
of a batch), each against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle.attention import attention_head, attention_step
from oracle.bf16 import bf16_bits_to_f64
from oracle.lmhead import lmhead_verify_step
from oracle.verify import verify_step
from paper_2402_11809_b200 import workloads
from test_gpu_parity import B, H, _check_verify, _small_cfg  # noqa: F401  (B, H: fixtures)

pytestmark = pytest.mark.gpu


# An odd vocabulary puts the rows at every element offset of the 16-byte grid; sizes around one vector, one
# sweep of a block (8192 bf16, 4096 f32 logits) and several chunks.
@pytest.mark.parametrize("mode", ["greedy", "sample", "literal", "filtered"])
@pytest.mark.parametrize("V,dtype", [(1, "bf16"), (7, "f32"), (9, "bf16"), (4095, "f32"), (8193, "bf16"), (16389, "f32"),
                                     (50257, "bf16")])
def test_verify_rows_off_the_16_byte_grid(B, H, mode, V, dtype):  # noqa: F811
    k, Bn = 3, 3
    cfg = _small_cfg(k, (5, 40), H_q=1, H_kv=1, d=64, Bn=Bn, V=V, dtype=dtype, seed=300 + V % 97)
    x = workloads.make_step_inputs(cfg)
    ctx = H.make_context(cfg, x)
    ds = H.DeviceStep(cfg, x)
    if mode == "greedy":
        ds.verify(ctx)
        _check_verify(ds, verify_step(x["logits"], x["cand"], x["cand_prob"], k, "greedy"), k)
        return
    resample = {"sample": "residual_pointmass", "literal": "paper_literal", "filtered": "residual_pointmass"}[mode]
    top_k = 5 if mode == "filtered" else 0
    v = ctx.verify_args(ds.logits, ds.cand, ds.cand_prob, ds.kv_len, ds.n_accept, ds.out_tokens, ds.n_out, ds.next_cand,
                        ds.next_cand_prob, ds.finished, k, mode=B.MODE_SAMPLE, temperature=0.9, seed=11,
                        resample=B.RESAMPLE_PAPER_LITERAL if mode == "literal" else B.RESAMPLE_RESIDUAL_POINTMASS,
                        seq_id=ds.seq_id, status=ds.status, top_k=top_k, top_p=0.9)
    ctx.space_verify(v)
    kw = dict(top_k=top_k, top_p=0.9) if top_k else {}
    r = verify_step(x["logits"], x["cand"], x["cand_prob"], k, "sample", temperature=0.9, seed=11, seq_id=x["seq_id"],
                    kv_len=x["kv_len"], resample=resample, **kw)
    _check_verify(ds, r, k, sample=True)


# Several segments per chunk (their lists are merged), chunks in both launches, and rows that defeat the
# expectation behind the bound: ascending logits (every later segment beats the list) and few distinct values.
@pytest.mark.parametrize("Bn,k,V,top_k,dtype", [(90, 2, 50003, 32, "bf16"), (2, 4, 20000, 32, "f32"), (1, 2, 8200, 3, "bf16"),
                                                (1, 2, 70001, 2, "f32"), (1, 5, 65537, 32, "f32")])
def test_filtered_sampling_on_sorted_and_tied_rows(B, H, Bn, k, V, top_k, dtype):  # noqa: F811
    cfg = _small_cfg(k, (5, 40), H_q=1, H_kv=1, d=64, Bn=Bn, V=V, dtype=dtype, seed=77)
    x = workloads.make_step_inputs(cfg)
    lf = np.sort(np.random.default_rng(3).standard_normal(V).astype(np.float32) * 2)
    even = np.round(lf[np.random.default_rng(4).permutation(V)])
    for b in range(Bn):
        row = lf if b % 2 else even
        x["logits"][b] = workloads.f32_to_bf16_bits(row) if dtype == "bf16" else row
        x["cand"][b] = V - 1 - np.arange(k) if b % 2 else np.argsort(-even, kind="stable")[:k]
    ctx = H.make_context(cfg, x)
    ds = H.DeviceStep(cfg, x)
    for resample, name in ((B.RESAMPLE_RESIDUAL_POINTMASS, "residual_pointmass"), (B.RESAMPLE_PAPER_LITERAL, "paper_literal")):
        ctx.space_verify(ctx.verify_args(ds.logits, ds.cand, ds.cand_prob, ds.kv_len, ds.n_accept, ds.out_tokens, ds.n_out,
                                         ds.next_cand, ds.next_cand_prob, ds.finished, k, mode=B.MODE_SAMPLE, seed=5,
                                         resample=resample, seq_id=ds.seq_id, top_k=top_k, top_p=1.0))
        r = verify_step(x["logits"], x["cand"], x["cand_prob"], k, "sample", temperature=1.0, seed=5, seq_id=x["seq_id"],
                        kv_len=x["kv_len"], resample=name, top_k=top_k, top_p=1.0)
        _check_verify(ds, r, k, sample=True)


# Wide batches by phase (target rows, then the mask rows of group i*): eight rows per sequence at k = 7, one mask
# row at k = 1, several groups of sequences, D and V off every tile, one box per range and several, a last stage of fewer
# slices taken first, and the last sequence's mask rows at the end of the hidden states.
@pytest.mark.parametrize("mode", ["greedy", "residual_pointmass", "paper_literal"])
@pytest.mark.parametrize("V,D,k,Bn", [(3001, 200, 7, 16), (131075, 264, 1, 67), (20000, 128, 5, 16), (129, 64, 5, 21), (40003, 136, 6, 18),
                                       (9001, 328, 7, 16)])
def test_lmhead_by_phase(B, H, mode, V, D, k, Bn):  # noqa: F811
    cfg = workloads.resolve_lmhead("lmhead_tiny", V=V, D=D, k=k, B=Bn, p_accept=(0.5, 1.0))
    x = workloads.make_lmhead_inputs(cfg)
    rng = np.random.default_rng(V)
    sample = mode != "greedy"
    if mode == "paper_literal":
        x["cand_prob"] = rng.uniform(0.05, 1.0, size=x["cand_prob"].shape).astype(np.float32)
    x["cand"][-1, -1] = V + 9                                # out of range: rejected, flagged
    kv_len = rng.integers(0, 3000, size=Bn).astype(np.int32)
    ctx = B.Context(max_batch=Bn, n_q_heads=8, n_kv_heads=8, head_dim=64, k_max=k, vocab=V, s_cap=256)
    i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")  # noqa: E731
    got = dict(n_accept=i32(Bn), out_tokens=i32(Bn, k + 1), n_out=i32(Bn), next_cand=i32(Bn, k),
               next_cand_prob=torch.full((Bn, k), float("nan"), device="cuda"),
               finished=torch.full((Bn,), 9, dtype=torch.uint8, device="cuda"))
    status = torch.zeros(Bn, dtype=torch.int32, device="cuda")
    keep = [H.to_dev(x[n]) for n in ("hidden", "weight", "cand", "cand_prob")] + [H.to_dev(kv_len)]
    a = ctx.lmhead_args(keep[0], keep[1], keep[2], k=k, eos_id=int(x["cand"][0, 0]), status=status, seed=7, temperature=0.9,
                        mode=B.MODE_SAMPLE if sample else B.MODE_GREEDY, cand_prob=keep[3], kv_len=keep[4],
                        resample=B.RESAMPLE_PAPER_LITERAL if mode == "paper_literal" else B.RESAMPLE_RESIDUAL_POINTMASS, **got)
    kw = dict(mode="sample", temperature=0.9, seed=7, kv_len=kv_len, resample=mode) if sample else {}
    r = lmhead_verify_step(x["hidden"], x["weight"], x["cand"], x["cand_prob"], k, eos_id=int(x["cand"][0, 0]), **kw)
    excl = np.zeros(Bn, bool)
    for b in range(Bn):
        i = int(r["n_accept"][b])
        used = [] if sample else [t * (k + 1) for t in range(k + 1)]
        used += [] if mode == "paper_literal" else [i * (k + 1) + o for o in range(1, k + 1)]
        excl[b] = bool(used) and r["row_gap"][b, used].min() <= 1e-3
    if sample:
        excl |= (r["accept_margin"] <= 1e-3).any(1) | (r["bonus_gap"] <= 1e-3) | (r["draft_gap"] <= 1e-3).any(1)
    assert excl.sum() <= max(1, Bn // 8)
    for again in range(2):                                   # counters and keys reset themselves
        n0 = ctx.launch_count
        ctx.space_lmhead_verify(a)
        assert (ctx.launch_count - n0) % 3 == 0              # targets, gather, masks per group of sequences
        h = {n: t.cpu().numpy() for n, t in got.items()}
        for n in ("n_accept", "out_tokens", "n_out", "next_cand", "finished"):
            assert np.array_equal(h[n][~excl], r[n][~excl]), (n, again)
        np.testing.assert_allclose(h["next_cand_prob"][~excl], r["next_cand_prob"][~excl], rtol=1e-3)
        assert status[-1].item() & B.ST_BAD_CANDIDATE and not status[:-1].any()


# Attention over at most one (sequence, kv head) per cluster: fewer tiles than pieces, first tiles that lie past the
# end or are the last, partial one, two query-row blocks per pair, lengths too unequal for the clustered cut (a long
# sequence next to short ones, at both kernels), and a sequence that does not fit.
@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("k,d,H_q,H_kv,lens", [
    (5, 128, 2, 2, (1, 90, 91, 92, 93, 700)), (2, 64, 4, 4, (0, 119, 120, 247, 1500)), (7, 128, 4, 2, (250, 300)),
    (4, 64, 8, 8, (1000,)), (3, 128, 2, 2, (9000, 40, 7)), (1, 64, 1, 1, (12000,)), (6, 64, 32, 4, (700, 905)),
    (4, 128, 16, 4, (30, 1500)), (4, 64, 8, 2, (9000, 5)), (6, 128, 16, 2, (2000,)),
])
def test_attention_clustered_cut(B, H, k, d, H_q, H_kv, lens, paged):  # noqa: F811
    cfg = _small_cfg(k, (min(lens), max(lens)), d=d, H_q=H_q, H_kv=H_kv, Bn=len(lens), V=64, seed=k)
    x = workloads.make_step_inputs(cfg, poison_tail=True)
    x["kv_len"][:] = lens
    rng = np.random.default_rng(1)
    for b, L in enumerate(lens):                             # keys for these lengths, the rest as poisoned as it was
        for name in ("k_cache", "v_cache"):
            x[name][b] = 0x7FC0
            x[name][b, :, : L + x["n_q"]] = workloads.f32_to_bf16_bits(rng.standard_normal((H_kv, L + x["n_q"], d), dtype=np.float32))
    y = workloads.to_pages(x) if paged else x
    y["kv_len"] = x["kv_len"].copy()
    if len(lens) > 2:
        y["kv_len"][1] = y["s_cap"]                          # does not fit: flagged, left alone
    ctx = H.make_context(cfg, y)
    ds = H.DeviceStep(cfg, y)
    for again in range(2):                                   # arrival counters reset themselves
        ds.out.fill_(float("nan"))
        ds.status.zero_()
        ds.attn(ctx)
        torch.cuda.synchronize()
        got, st = ds.out.cpu().numpy().astype(np.float64), ds.status.cpu().numpy()
        for b, L in enumerate(lens):
            if y["kv_len"][b] != L:
                assert st[b] == B.ST_CAPACITY and np.isnan(got[b]).all()
                continue
            assert st[b] == 0
            ref, lse = attention_step(x["q"][b:b + 1], x["k_cache"][b:b + 1], x["v_cache"][b:b + 1], x["kv_len"][b:b + 1], k, x["scale"])
            H.check_attention(got[b:b + 1], ref, f"sequence {b} of length {L}")
            np.testing.assert_allclose(ds.lse[b].cpu().numpy(), lse[0], rtol=0, atol=2e-3)


# A page's tail rows are cleared while the V ring is several rounds in (head size 64: four V stages, three S buffers).
@pytest.mark.parametrize("d", [64, 128])
def test_rows_kernel_long_paged_shares(B, H, d):  # noqa: F811
    k, H_q, H_kv = 4, 8, 2
    cfg = _small_cfg(k, (2300, 2350), d=d, H_q=H_q, H_kv=H_kv, Bn=80, V=64, seed=3)     # more pairs than blocks: long shares
    x = workloads.to_pages(workloads.make_step_inputs(cfg))
    ctx = H.make_context(cfg, x)
    ds = H.DeviceStep(cfg, x)
    ds.attn(ctx)
    torch.cuda.synchronize()
    assert not ds.status.any()
    assert torch.isfinite(ds.out).all()
    c = workloads.make_step_inputs(cfg)
    for b in (0, 41, 79):
        ref, _ = attention_step(c["q"][b:b + 1], c["k_cache"][b:b + 1], c["v_cache"][b:b + 1], c["kv_len"][b:b + 1], k, c["scale"])
        H.check_attention(ds.out[b:b + 1].cpu().numpy().astype(np.float64), ref, f"sequence {b}")


# space_step_host reaches into pinned buffers by kernels and copies pageable or misaligned ones; one sequence does
# not fit its cache and is left alone.  V = 40001: the verification takes two launches over PCIe.
@pytest.mark.parametrize("V", [501, 40001])
@pytest.mark.parametrize("where", ["pinned", "pageable", "misaligned"])
def test_host_step_transfers(B, H, where, V):  # noqa: F811
    k, Bn, H_q, H_kv, d = 3, 3, 4, 2, 64
    cfg = workloads.resolve("tiny", B=Bn, H_q=H_q, H_kv=H_kv, d=d, L=(20, 140), k=k, V=V, logits_dtype="bf16", seed=5)
    x = workloads.make_step_inputs(cfg)
    n_q, cap = x["n_q"], x["s_cap"]
    x["kv_len"][1] = cap - n_q + 1                           # one row too many
    ctx = B.Context(max_batch=Bn, n_q_heads=H_q, n_kv_heads=H_kv, head_dim=d, k_max=k, vocab=V, host_staging=1, s_cap=cap)

    def host(a):
        a = a.view(np.int16) if a.dtype == np.uint16 else a
        flat = torch.zeros(a.size + 1, dtype=torch.from_numpy(a).dtype, pin_memory=where != "pageable")
        t = flat[1:] if where == "misaligned" else flat[:-1]
        return t.view(a.shape).copy_(torch.from_numpy(a))

    z = lambda *s, dt=torch.int32: torch.zeros(s, dtype=dt)  # noqa: E731
    r = verify_step(x["logits"], x["cand"], x["cand_prob"], k, "greedy")
    for resident in (0, 1, 1):
        h = {n: host(x[n]) for n in ("q", "k_cache", "v_cache", "logits", "cand", "cand_prob", "kv_len")}
        h.update(out=host(np.zeros((Bn, n_q, H_q, d), np.float32)), n_accept=z(Bn), out_tokens=z(Bn, k + 1), n_out=z(Bn),
                 next_cand=z(Bn, k), next_cand_prob=z(Bn, k, dt=torch.float32), finished=z(Bn, dt=torch.uint8), status=z(Bn))
        ctx.space_step_host(B.HostStepArgs(batch=Bn, k=k, vocab=V, logits_dtype=B.DTYPE_BF16, mode=B.MODE_GREEDY, eos_id=-1,
                                           scale=x["scale"], temperature=1.0, cache_resident=resident,
                                           **{n: t.data_ptr() for n, t in h.items()}))
        assert h["status"].tolist() == [0, B.ST_CAPACITY, 0]
        for n in ("n_accept", "out_tokens", "n_out", "next_cand"):
            assert np.array_equal(h[n].numpy(), r[n]), (n, resident)
        for b in (0, 2):
            L, na = int(x["kv_len"][b]), int(r["n_accept"][b])
            ref, _ = attention_step(x["q"][b:b + 1], x["k_cache"][b:b + 1], x["v_cache"][b:b + 1], x["kv_len"][b:b + 1], k, x["scale"])
            H.check_attention(h["out"][b:b + 1].numpy().astype(np.float64), ref, where)
            assert int(h["kv_len"][b]) == L + na + 1
            for name in ("k_cache", "v_cache"):
                got = h[name].numpy().view(np.uint16)[b]
                for g in range(na + 1):
                    assert np.array_equal(got[:, L + g], x[name][b][:, L + g * (k + 1)])
        assert np.array_equal(h["k_cache"].numpy().view(np.uint16)[1], x["k_cache"][1])


def _growing_keys(x, G, per_tile):
    """Adds t * (a multiple of the signs of block row 0's query) to the keys of tile t of every kv head, so that the scores
    of that row grow by per_tile binary orders of magnitude from tile to tile.  Returns the least amount by which a tile
    exceeds the first key of one at least two tiles before it."""
    kf, qf = (bf16_bits_to_f64(x[n]).astype(np.float32) for n in ("k_cache", "q"))
    tile = np.arange(kf.shape[2]) // 128
    log2e, least = float(np.log2(np.e)), np.inf
    for b in range(kf.shape[0]):
        for h in range(kf.shape[1]):
            q = qf[b, 0, h * G]
            kf[b, h] += tile[:, None] * np.sign(q) * np.float32(per_tile / (log2e * x["scale"] * np.abs(q).sum()))
    x["k_cache"] = workloads.f32_to_bf16_bits(kf)
    kf = bf16_bits_to_f64(x["k_cache"])
    for b in range(kf.shape[0]):
        L = int(x["kv_len"][b])                              # (cached keys: every row sees them)
        for h in range(kf.shape[1]):
            s = kf[b, h, :L] @ qf[b, 0, h * G].astype(np.float64) * (x["scale"] * log2e)
            top = [s[t:t + 128].max() for t in range(0, L, 128)]
            least = min([least] + [top[t] - s[u * 128] for t in range(2, len(top)) for u in range(t - 1)])
    return least


# Every width of the transposed attention kernel (16, 32, 48, 64 padded query rows) with several tiles per block, so
# that its rings of scores, P and tiles come round, clustered (two sequences) and in the flat cut (more pairs than
# SMs).  With keys whose scores grow along the sequence every share has a tile that exceeds its reference by more than
# 2^60, and the references move in its middle (the rows kernel takes the same inputs).
@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("per_tile", [0, 40])
@pytest.mark.parametrize("k,G,d,Bn,H_kv", [(1, 1, 64, 2, 12), (2, 1, 128, 40, 4), (3, 1, 128, 2, 12), (3, 2, 64, 2, 12),
                                           (4, 1, 128, 2, 12), (5, 1, 128, 2, 12), (5, 1, 64, 40, 4), (7, 1, 128, 2, 12),
                                           (7, 1, 64, 2, 12), (6, 1, 128, 40, 4)])
def test_transposed_kernel_widths(B, H, k, G, d, Bn, H_kv, per_tile, paged):  # noqa: F811
    cfg = _small_cfg(k, (700, 3100 if Bn == 2 else 900), d=d, H_q=H_kv * G, H_kv=H_kv, Bn=Bn, V=64, seed=k + d)
    x = workloads.make_step_inputs(cfg)
    if per_tile:
        assert _growing_keys(x, G, per_tile) > 60
        # two sequences: at most 148 // 24 = 6 pieces per pair, taking every sixth tile; otherwise a block's share is
        # longer than a pair
        assert x["kv_len"].max() // 128 > (7 if Bn == 2 else 5)
    y = workloads.to_pages(x) if paged else x
    ctx = H.make_context(cfg, y)
    for impl in (B.ATTN_TENSOR, B.ATTN_TENSOR_ROWS)[:2 if per_tile else 1]:
        ds = H.DeviceStep(cfg, y)
        ds.attn(ctx, impl=impl)
        assert not ds.status.any()
        got = ds.out.cpu().numpy().astype(np.float64)
        for b in (0, Bn - 1):                                # first and last pairs of the cut
            for h in (0, H_kv * G - 1):
                ref, _ = attention_head(x["q"][b, :, h], x["k_cache"][b, h // G], x["v_cache"][b, h // G], int(x["kv_len"][b]), k, x["scale"])
                H.check_attention(got[b:b + 1, :, h], ref[None], f"sequence {b} head {h}")


# Projection with the tokens on the M extent: few rows and 129..176 padded ones, ranges of one box and of two, a last
# box of one accumulator, D off the slices, odd vocabularies; next to widths that keep the rows on M.  Sampling: noise
# from the table and past its end (many noisy rows), sequence ids and positions per row.
@pytest.mark.parametrize("mode", ["greedy", "residual_pointmass", "paper_literal"])
@pytest.mark.parametrize("V,D,k,Bn", [(30011, 72, 2, 1), (29000, 136, 5, 1), (40003, 64, 7, 1), (38001, 200, 5, 4), (50257, 64, 3, 11),
                                      (57003, 72, 1, 40), (32000, 64, 3, 15), (60001, 64, 1, 25), (400, 64, 5, 2)])
def test_lmhead_orientations(B, H, mode, V, D, k, Bn):  # noqa: F811
    cfg = workloads.resolve_lmhead("lmhead_tiny", V=V, D=D, k=k, B=Bn, p_accept=(0.5, 1.0))
    x = workloads.make_lmhead_inputs(cfg)
    rng = np.random.default_rng(V)
    sample = mode != "greedy"
    if mode == "paper_literal":
        x["cand_prob"] = rng.uniform(0.05, 1.0, size=x["cand_prob"].shape).astype(np.float32)
    kv_len = rng.integers(0, 3000, size=Bn).astype(np.int32)
    ctx = B.Context(max_batch=Bn, n_q_heads=8, n_kv_heads=8, head_dim=64, k_max=k, vocab=V, s_cap=256)
    i32 = lambda *s: torch.empty(s, dtype=torch.int32, device="cuda")  # noqa: E731
    got = dict(n_accept=i32(Bn), out_tokens=i32(Bn, k + 1), n_out=i32(Bn), next_cand=i32(Bn, k),
               next_cand_prob=torch.empty((Bn, k), device="cuda"), finished=torch.empty((Bn,), dtype=torch.uint8, device="cuda"))
    keep = [H.to_dev(x[n]) for n in ("hidden", "weight", "cand", "cand_prob")] + [H.to_dev(kv_len)]
    a = ctx.lmhead_args(keep[0], keep[1], keep[2], k=k, eos_id=-1, seed=7, temperature=0.9,
                        mode=B.MODE_SAMPLE if sample else B.MODE_GREEDY, cand_prob=keep[3], kv_len=keep[4],
                        resample=B.RESAMPLE_PAPER_LITERAL if mode == "paper_literal" else B.RESAMPLE_RESIDUAL_POINTMASS, **got)
    kw = dict(mode="sample", temperature=0.9, seed=7, kv_len=kv_len, resample=mode) if sample else {}
    r = lmhead_verify_step(x["hidden"], x["weight"], x["cand"], x["cand_prob"], k, eos_id=-1, **kw)
    excl = np.zeros(Bn, bool)                                # decisions inside the tie bands of the by-phase test
    for b in range(Bn):
        i = int(r["n_accept"][b])
        used = [] if sample else [t * (k + 1) for t in range(k + 1)]
        used += [] if mode == "paper_literal" else [i * (k + 1) + o for o in range(1, k + 1)]
        excl[b] = bool(used) and r["row_gap"][b, used].min() <= 1e-3
    if sample:
        excl |= (r["accept_margin"] <= 1e-3).any(1) | (r["bonus_gap"] <= 1e-3) | (r["draft_gap"] <= 1e-3).any(1)
    assert excl.sum() <= Bn // 8                             # (none of a few: something is left to compare)
    for again in range(2):
        for n, t in got.items():                             # (a call that wrote nothing does not pass)
            t.fill_({"next_cand_prob": float("nan"), "finished": 9}.get(n, -7))
        ctx.space_lmhead_verify(a)
        h = {n: t.cpu().numpy() for n, t in got.items()}
        for n in ("n_accept", "out_tokens", "n_out", "next_cand", "finished"):
            assert np.array_equal(h[n][~excl], r[n][~excl]), (n, again)
        np.testing.assert_allclose(h["next_cand_prob"][~excl], r["next_cand_prob"][~excl], rtol=1e-3)


# The single-launch greedy verify moves its slice of the rows to commit while it scans, one 16-byte piece per thread,
# where that covers them all (not for k = 1 with many heads and a short vocabulary), and after the scan otherwise
# (also with rows off the 16-byte grid).
@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("k,H_kv,d,V,Bn", [(1, 32, 128, 704, 3), (1, 32, 128, 20000, 2), (7, 1, 64, 48, 3), (5, 8, 64, 9000, 2), (5, 8, 64, 9001, 2)])
def test_commit_under_the_scan(B, H, k, H_kv, d, V, Bn, paged):  # noqa: F811
    from oracle.commit import commit_step
    cfg = _small_cfg(k, (100, 400), d=d, H_q=H_kv, H_kv=H_kv, Bn=Bn, V=V, seed=V)
    x = workloads.make_step_inputs(cfg)
    for i in range(k):                                       # the first sequence accepts every candidate
        x["logits"][0, i * (k + 1), x["cand"][0, i]] = workloads.f32_to_bf16_bits(np.float32([40.0]))[0]
    y = workloads.to_pages(x) if paged else x
    ctx = H.make_context(cfg, y)
    ds = H.DeviceStep(cfg, y)
    ds.verify_commit(ctx)
    r = verify_step(x["logits"], x["cand"], x["cand_prob"], k, "greedy")
    assert not _check_verify(ds, r, k).any() and r["n_accept"][0] == k
    new_len, _, _ = commit_step(x["k_cache"], x["v_cache"], x["kv_len"], r["n_accept"], k)      # (in place)
    assert np.array_equal(ds.kv_len_out.cpu().numpy(), new_len)
    for name, dev in (("k_cache", ds.k_cache), ("v_cache", ds.v_cache)):
        got = H.bf16_to_bits(dev)
        for b in range(Bn):
            n = int(new_len[b])
            if paged:
                rows = np.concatenate([got[pg] for pg in y["page_table"][b][: -(-n // 128)]], axis=1)
            else:
                rows = got[b]
            assert np.array_equal(rows[:, :n], x[name][b][:, :n]), (name, b)


# Filtered sampling on both sides of the line between one launch over all block rows and two (few rows: 30 MB of
# logits, 110 rows; more rows: 16 MB; rows off the 16-byte grid; blocks that do not fit at once), with the commit on board: the same decisions and cache either way.
@pytest.mark.parametrize("Bn,k,V,dtype,launches", [(3, 5, 128256, "bf16", 1), (2, 4, 128256, "f32", 1), (4, 5, 64064, "bf16", 2),
                                                  (3, 5, 146000, "bf16", 2), (7, 3, 70001, "bf16", 1),
                                                  (2, 6, 50257, "f32", 2), (12, 2, 50257, "f32", 1), (3, 4, 100000, "f32", 2),
                                                  (1, 7, 80001, "f32", 2), (2, 4, 128257, "f32", 1)])
def test_filtered_one_launch_or_two(B, H, Bn, k, V, dtype, launches):  # noqa: F811
    from oracle.commit import commit_step
    cfg = workloads.resolve("sampling64", B=Bn, H_q=2, H_kv=2, d=64, L=(5, 200), k=k, V=V, logits_dtype=dtype, seed=V % 89)
    x = workloads.make_step_inputs(cfg)
    ctx = H.make_context(cfg, x)
    ds = H.DeviceStep(cfg, x)
    v = ctx.verify_args(ds.logits, ds.cand, ds.cand_prob, ds.kv_len, ds.n_accept, ds.out_tokens, ds.n_out, ds.next_cand,
                        ds.next_cand_prob, ds.finished, k, mode=B.MODE_SAMPLE, temperature=0.9, seed=3, seq_id=ds.seq_id,
                        status=ds.status, top_k=10, top_p=0.95)
    n0 = ctx.launch_count
    ctx.space_verify_commit(v, ctx.commit_args(ds.k_cache, ds.v_cache, ds.n_accept, ds.kv_len, k, kv_len_out=ds.kv_len_out))
    assert ctx.launch_count - n0 == launches
    r = verify_step(x["logits"], x["cand"], x["cand_prob"], k, "sample", temperature=0.9, seed=3, seq_id=x["seq_id"],
                    kv_len=x["kv_len"], top_k=10, top_p=0.95)
    assert not _check_verify(ds, r, k, sample=True).any()
    new_len, _, _ = commit_step(x["k_cache"], x["v_cache"], x["kv_len"], r["n_accept"], k)       # (in place)
    assert np.array_equal(ds.kv_len_out.cpu().numpy(), new_len)
    assert np.array_equal(H.bf16_to_bits(ds.k_cache), x["k_cache"]) and np.array_equal(H.bf16_to_bits(ds.v_cache), x["v_cache"])


# Clusters launched for lengths that are too unequal (or too long for the pieces a cluster can hold) for them: every cut of
# the list over the grid is combined by the whole cluster of the block that finds its last piece.  Four row blocks of one
# pair over all blocks, two pairs of a smaller head, one long sequence among short ones, two row blocks of the transposed
# kernel.  Twice: the counters are back where they were, and the pieces are added in a fixed order.
@pytest.mark.parametrize("k,d,H_q,H_kv,lens,paged,row_blocks", [(6, 128, 8, 1, (9000,), False, 4), (6, 64, 16, 2, (9001,), True, 4),
                                                                (5, 64, 4, 4, (16000, 800, 127, 640, 0), False, 1),
                                                                (7, 128, 2, 1, (16000, 300), True, 2)])
def test_attention_cuts_combined_by_the_cluster(B, H, k, d, H_q, H_kv, lens, paged, row_blocks):  # noqa: F811
    # These lengths do not get the clustered cut, whatever number of pieces is launched: its longest piece has more than ten
    # tiles over an even share (plan_clusters, cluster_fits; up to two clusters fewer than the SMs would hold may fit).
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles, pairs = [-(-(L + (k + 1) ** 2) // 128) for L in lens], len(lens) * H_kv
    launched = [c for c in range(1, 16 // row_blocks + 1) if pairs * c * row_blocks <= sms]
    for c in launched:
        groups = max(pairs, sms // (c * row_blocks) - 2) * c
        assert -(-max(tiles) // c) > -(-sum(tiles) * H_kv // groups) + 10, c
    cfg = _small_cfg(k, (0, max(lens)), d=d, H_q=H_q, H_kv=H_kv, Bn=len(lens), V=64, seed=k + d + len(lens))
    x = workloads.make_step_inputs(cfg)
    x["kv_len"][:] = lens
    y = workloads.to_pages(x) if paged else x
    ctx = H.make_context(cfg, y)
    ds = H.DeviceStep(cfg, y)
    n0 = ctx.launch_count
    ds.attn(ctx)
    assert ctx.launch_count - n0 == 1 and not ds.status.any()    # (no merge kernel)
    got, got_lse = ds.out.clone(), ds.lse.clone()
    ds.out.fill_(float("nan"))
    ds.lse.fill_(float("nan"))
    ds.attn(ctx)
    assert torch.equal(got, ds.out) and torch.equal(got_lse, ds.lse)
    got, got_lse = got.cpu().numpy().astype(np.float64), got_lse.cpu().numpy()
    for b, L in enumerate(lens):
        for h in (0, H_q - 1):
            G = H_q // H_kv
            ref, lse = attention_head(x["q"][b, :, h], x["k_cache"][b, h // G], x["v_cache"][b, h // G], L, k, x["scale"])
            H.check_attention(got[b:b + 1, :, h], ref[None], f"sequence {b} head {h}")
            np.testing.assert_allclose(got_lse[b, h], lse, rtol=0, atol=2e-3)


# Sweeps of a block that lie in its chunk as a whole and the one that does not, at the edges (a sweep is 8192 bf16 or 4096
# f32 logits), in launches of more blocks than three per SM hold (576 and 640 of one chunk), with the commit on board; and
# the two launches of sampling.
@pytest.mark.parametrize("V,dtype", [(296, "bf16"), (8192, "bf16"), (8200, "bf16"), (16380, "bf16"), (24584, "bf16"),
                                     (4096, "f32"), (4100, "f32"), (12284, "f32")])
@pytest.mark.parametrize("mode,Bn,k,paged", [("greedy", 16, 5, False), ("greedy", 40, 3, True), ("sample", 3, 4, False)])
def test_verify_sweeps_and_many_blocks(B, H, mode, Bn, k, paged, V, dtype):  # noqa: F811
    from oracle.commit import commit_step
    cfg = _small_cfg(k, (5, 150), H_q=2, H_kv=2, d=64, Bn=Bn, V=V, dtype=dtype, seed=V % 97 + Bn)
    x = workloads.make_step_inputs(cfg)
    y = workloads.to_pages(x) if paged else x
    ctx = H.make_context(cfg, y)
    ds = H.DeviceStep(cfg, y)
    if mode == "sample":
        v = ctx.verify_args(ds.logits, ds.cand, ds.cand_prob, ds.kv_len, ds.n_accept, ds.out_tokens, ds.n_out, ds.next_cand,
                            ds.next_cand_prob, ds.finished, k, mode=B.MODE_SAMPLE, temperature=0.9, seed=5, seq_id=ds.seq_id,
                            status=ds.status)
        ctx.space_verify(v)
        r = verify_step(x["logits"], x["cand"], x["cand_prob"], k, "sample", temperature=0.9, seed=5, seq_id=x["seq_id"],
                        kv_len=x["kv_len"])
        assert _check_verify(ds, r, k, sample=True).sum() <= 1
        return
    ds.verify_commit(ctx)
    r = verify_step(x["logits"], x["cand"], x["cand_prob"], k, "greedy")
    assert not _check_verify(ds, r, k).any()
    new_len, _, _ = commit_step(x["k_cache"], x["v_cache"], x["kv_len"], r["n_accept"], k)       # (in place)
    assert np.array_equal(ds.kv_len_out.cpu().numpy(), new_len)
    got = H.bf16_to_bits(ds.k_cache)
    for b in range(Bn):
        rows = np.concatenate([got[pg] for pg in y["page_table"][b][: -(-int(new_len[b]) // 128)]], axis=1) if paged else got[b]
        assert np.array_equal(rows[:, :int(new_len[b])], x["k_cache"][b][:, :int(new_len[b])]), b


# Sampling by phase: target row i* is projected once more beside the mask rows and draws the extra token there.  As many
# rows as an accumulator holds, groups of sequences with a small last one, a range of two boxes.
@pytest.mark.parametrize("mode", ["residual_pointmass", "paper_literal"])
@pytest.mark.parametrize("V,D,k,Bn", [(9001, 64, 7, 17), (9000, 72, 4, 50), (40009, 64, 5, 42)])
def test_lmhead_extra_token_in_the_second_pass(B, H, mode, V, D, k, Bn):  # noqa: F811
    test_lmhead_orientations(B, H, mode, V, D, k, Bn)


# Hidden rows as wide as the gathered rows' buffer takes for a full accumulator, and wider.
@pytest.mark.parametrize("mode", ["greedy", "residual_pointmass"])
@pytest.mark.parametrize("V,D,k,Bn", [(2101, 16384, 5, 12), (1501, 24008, 1, 65)])
def test_lmhead_by_phase_wide_hidden_rows(B, H, mode, V, D, k, Bn):  # noqa: F811
    test_lmhead_by_phase(B, H, mode, V, D, k, Bn)
