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
