"""The standalone gate, which splits the fp32 gate rows itself (staged by TMA up
to 32 rows, loaded to registers beyond; one group of at most 16 experts with
Top-1 is decided from registers), against the layer call, which takes prepared
rows: the same sums in the same order, so the same bits.  Gate rows at the edges
of the variants, d_model that ends inside a 64-column stage, one CTA and two per
tile, ragged token tiles, and rows and experts without a finite logit."""

import pytest
import torch

from paper_2508_06024_gb300 import build as B
from paper_2508_06024_gb300 import ec2moe as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    C.load()


@pytest.mark.parametrize("E,K,k,renorm", [(1, 1, 1, 1), (16, 1, 1, 0), (15, 1, 2, 1), (17, 1, 1, 1), (14, 2, 1, 0),
                                          (24, 8, 3, 0), (32, 1, 4, 0), (33, 1, 1, 0)])
@pytest.mark.parametrize("d", [96, 800, 2080])
def test_standalone_gate_equals_layer_gate(E, K, k, renorm, d):
    T, f = 300, 32
    g = torch.Generator(device="cuda")
    g.manual_seed(E * 100 + d)

    def normal(*shape, dtype=torch.float32):
        return torch.randn(*shape, generator=g, device="cuda").to(dtype)

    X = normal(T, d, dtype=torch.bfloat16)
    X[5] = float("nan")
    X[T - 1] = float("inf")
    t = dict(W_local=normal(E, d) / d ** 0.5, b_local=normal(E), W1=normal(E, f, d, dtype=torch.bfloat16),
             W3=normal(E, f, d, dtype=torch.bfloat16), W2=normal(E, d, f, dtype=torch.bfloat16))
    if K > 1:
        t.update(W_global=normal(K, d) / d ** 0.5, b_global=normal(K))
    if E > 3:
        t["b_local"][3] = float("-inf")
    mask = torch.ones(E, dtype=torch.uint8)
    if E > 8:
        mask[0] = mask[E // 2] = 0
    mask = C.host_mask(mask)
    desc = C.make_desc(T=T, d=d, E=E, d_ff=f, k=k, n_groups=K, act=C.SWIGLU, dtype=C.BF16, renorm_topk=renorm)

    def empty(*shape, dtype):
        return torch.empty(*shape, dtype=dtype, device="cuda")

    got = [empty(T, k, dtype=torch.int32), empty(T, k, dtype=torch.float32)]
    ref = [empty(T, k, dtype=torch.int32), empty(T, k, dtype=torch.float32)]
    C.ec2moe_gate(desc, X, t["W_local"], t["b_local"], t.get("W_global"), t.get("b_global"), mask, *got)
    ws = empty(C.ec2moe_workspace_size(desc), dtype=torch.uint8)
    C.ec2moe_layer_forward(desc, C.make_weights(**t), X, mask, empty(T, d, dtype=torch.bfloat16), *ref,
                           empty(E, dtype=torch.int32), None, ws, ws.numel())
    assert C.ec2moe_last_device_error() == C.OK
    assert torch.equal(got[0], ref[0])
    assert torch.allclose(got[1], ref[1], rtol=0.0, atol=0.0, equal_nan=True)
