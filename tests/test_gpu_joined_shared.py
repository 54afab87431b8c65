"""Shared experts as further groups of the routed experts' two launches: the
layer against the chain of single entry points, which runs them in launches of
their own, bit for bit (the same sums in the same order), on each GEMM kernel
that takes them: tokens on M (single CTAs and pairs) and tokens on N, for the up
and the down projection."""

import pytest
import torch

from paper_2508_06024_gb300 import build as B
from paper_2508_06024_gb300 import ec2moe as C
from paper_2508_06024_gb300 import synth as S
from paper_2508_06024_gb300.runner import LayerRun, desc_for
from tests.parity import gemm_launches

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    C.load()


# 18 rows (the first size past the swapped-operand kernel), a ragged decode
# batch, tokens on N for the up projection (K = 2048, 667 expected rows per group;
# the down projection's K = 1408 stays on M), pairs, three shared experts of GELU
# in a Top-1 layer; tokens on N for both projections (K >= 2048, d_ff not a
# multiple of 64, 400 and 360 expected rows per group).  The last column: launches
# of the tokens-on-N kernel.
@pytest.mark.parametrize("cfg,tok", [
    (S.preset("finegrained_bf16", T=3, seed=81), 0),
    (S.preset("finegrained_bf16", T=77, seed=82), 0),
    (S.preset("finegrained_bf16", T=2001, E=16, n_allowed=16, n_groups=2, seed=83), 1),
    (S.preset("finegrained_bf16", T=4096, E=8, n_allowed=8, n_groups=2, zipf_s=0.0, seed=84), 0),
    (S.preset("switch_bf16", T=500, d_ff=512, n_shared=3, d_ff_shared=512, seed=85), 0),
    (S.preset("finegrained_bf16", T=1000, E=8, n_allowed=8, n_groups=2, k=2, d_ff=2080, d_ff_shared=2080, seed=86), 2),
    (S.preset("switch_bf16", T=901, d=2048, E=4, n_allowed=4, d_ff=2080, n_shared=1, d_ff_shared=2080, seed=87), 2)],
    ids=["first-size", "ragged", "tokens-on-n-up", "pairs", "gelu-top1", "tokens-on-n", "tokens-on-n-gelu"])
def test_joined_equals_separate(cfg, tok):
    inp = S.make_inputs(cfg, device="cuda")
    run = LayerRun(cfg, inp)
    assert gemm_launches(run.forward, "tok_gemm_kernel") in (tok, None)
    y = run.forward()
    assert C.ec2moe_last_device_error() == C.OK
    desc, T, k, d = desc_for(cfg), cfg.T, cfg.k, cfg.d
    n, bf = T * k, torch.bfloat16
    dev = dict(device="cuda")
    i32 = dict(dtype=torch.int32, **dev)
    xh, xp = torch.empty(T, d, dtype=bf, **dev), torch.empty(n, d, dtype=bf, **dev)
    slot, sh = torch.empty(n, d, dtype=bf, **dev), torch.empty(cfg.n_shared * T, d, dtype=bf, **dev)
    counts, offsets, perm = torch.empty(cfg.E, **i32), torch.empty(cfg.E + 1, **i32), torch.empty(n, **i32)
    wr = torch.empty(C.ec2moe_route_workspace_size(desc), dtype=torch.uint8, **dev)
    ws = torch.empty(C.ec2moe_experts_workspace_size(desc), dtype=torch.uint8, **dev)
    y2 = torch.empty_like(y)
    C.ec2moe_lr_decode(desc, run.Z, inp["V_dec"], xh)
    C.ec2moe_route(desc, run.topk_idx, counts, offsets, perm, None, xh, d, xp, wr, wr.numel())
    C.ec2moe_experts(desc, xp, offsets, inp["W1"], inp["W3"], inp["W2"], run.topk_w, perm, slot, ws, ws.numel())
    C.ec2moe_shared_experts(desc, xh, inp["W1s"], inp["W3s"], inp["W2s"], sh, ws, ws.numel())
    C.ec2moe_combine(desc, slot, sh, y2)
    assert C.ec2moe_last_device_error() == C.OK
    assert torch.equal(y, y2)
