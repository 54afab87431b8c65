"""The combine of split-K expert outputs (at most 128 routed rows, d_ff >= 4096)
through the layer call against the oracle, at the edges of its split: rows of
d_model that are not a multiple of a block's 64 eight-column chunks (4 chunks
and 60 chunks in the last block), slots times K ranges that are not a multiple
of the eight loads in flight, one to eight slots, shared experts.  The layer
runs twice: the second pass finds the first one's sums in the workspace."""

import numpy as np
import pytest
import torch

from oracle import ec2moe_oracle as orc
from paper_2508_06024_gb300 import build as B
from paper_2508_06024_gb300 import ec2moe as C
from paper_2508_06024_gb300 import synth as S
from paper_2508_06024_gb300.runner import LayerRun
from tests.parity import TIE_GAP, oracle_inputs, output_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    C.load()


@pytest.mark.parametrize("cfg", [
    S.preset("decode_bf16", T=1, k=1, d=1056, d_ff=4096, n_allowed=4, r=128, seed=91),
    S.preset("decode_bf16", T=5, k=3, d=992, d_ff=4096, n_allowed=8, r=128, n_shared=2, d_ff_shared=512, seed=92),
    S.preset("decode_bf16", T=16, k=8, d=1056, d_ff=4096, n_allowed=8, r=0, seed=93),
    S.preset("decode_bf16", T=25, k=5, d=512, d_ff=4608, n_allowed=8, r=128, n_shared=1, d_ff_shared=512, seed=94)],
    ids=lambda c: f"T{c.T}-k{c.k}-d{c.d}-shared{c.n_shared}")
def test_split_k_combine(cfg):
    inp = S.make_inputs(cfg, device="cuda")
    run = LayerRun(cfg, inp)
    first = run.forward().clone()
    y = run.forward()
    assert C.ec2moe_last_device_error() == C.OK
    assert torch.equal(first, y)
    ref = orc.layer_forward(oracle_inputs(inp, lazy_experts=True), cfg.n_groups, cfg.k, cfg.act, bool(cfg.renorm_topk))
    keep = ref["gap_boundary"] >= TIE_GAP
    assert keep.any()
    output_check(y.double().cpu().numpy()[np.flatnonzero(keep)], ref["y"][keep], True)
