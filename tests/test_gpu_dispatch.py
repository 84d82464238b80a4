"""GPU parity at the edges of the kernels' dispatch rules (row alignment, chunk and tile remainders, grouping
of a batch), each against the fp64 oracle."""
import numpy as np
import pytest
import torch

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
@pytest.mark.parametrize("Bn,k,V,top_k,dtype", [(90, 2, 50003, 32, "bf16"), (2, 4, 20000, 32, "f32"), (1, 2, 8200, 3, "bf16")])
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
