"""The expert GEMM with the tokens on the MMA's N side (groups of a few hundred
rows, long K), through ec2moe_experts on hand-built group layouts: one row, one
past a tile's padding, a group over several tiles, an empty group, and widths
that end inside a weight block.

The reference multiplies the stored bf16 values in fp32 and rounds the hidden
rows to bf16 as the kernel does; what differs is the fp32 order of the sums,
which can move a rounding of a hidden or output value by one bf16 step (2^-8),
so the bounds are those of every bf16 output (relative Frobenius 1e-2).
"""

import pytest
import torch

from paper_2508_06024_gb300 import build as B
from paper_2508_06024_gb300 import ec2moe as C
from tests.parity import gemm_launches, rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    C.load()


def _case(rows, d, ff, act, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def normal(*shape, fan_in):
        return (torch.randn(*shape, generator=g, device="cuda") / fan_in ** 0.5).bfloat16()

    E, n = len(rows), sum(rows)
    t = dict(X=normal(n, d, fan_in=1), W1=normal(E, ff, d, fan_in=d), W3=normal(E, ff, d, fan_in=d),
             W2=normal(E, d, ff, fan_in=ff), w=torch.rand(n, generator=g, device="cuda"),
             perm=torch.randperm(n, generator=g, device="cuda").int())
    off = [sum(rows[:i]) for i in range(E + 1)]
    desc = C.make_desc(T=n, d=d, E=E, d_ff=ff, k=1, act=act, dtype=C.BF16)
    ws = torch.empty(C.ec2moe_experts_workspace_size(desc), dtype=torch.uint8, device="cuda")
    return t, off, desc, ws


def _run(t, off, desc, ws):
    out = torch.full((desc.T, desc.d), float("nan"), device="cuda").bfloat16()
    C.ec2moe_experts(desc, t["X"], torch.tensor(off, dtype=torch.int32, device="cuda"), t["W1"], t["W3"], t["W2"], t["w"],
                     t["perm"], out, ws, ws.numel())
    return out


def _check_group(t, e, lo, hi, act, out):
    x = t["X"][lo:hi].float()
    u = x @ t["W1"][e].float().T
    h = torch.nn.functional.gelu(u) if act == C.GELU else torch.nn.functional.silu(u) * (x @ t["W3"][e].float().T)
    p = t["perm"][lo:hi].long()
    ref = (h.bfloat16().float() @ t["W2"][e].float().T) * t["w"][p][:, None]
    assert rel_fro(out[p].double().cpu().numpy(), ref.double().cpu().numpy()) <= 1e-2


@pytest.mark.parametrize("act,ff", [(C.SWIGLU, 2464), (C.GELU, 4896)], ids=["swiglu", "gelu"])
@pytest.mark.parametrize("rows", [[1, 257, 0, 800], [33, 256, 511, 288]], ids=["uneven", "edges"])
def test_experts_tokens_on_n(rows, act, ff):
    t, off, desc, ws = _case(rows, 2592, ff, act, 7)
    assert gemm_launches(lambda: _run(t, off, desc, ws), "tok_gemm_kernel") in (2, None)
    out = _run(t, off, desc, ws)
    assert C.ec2moe_last_device_error() == C.OK
    assert not bool(out.isnan().any())
    for e in range(len(rows)):
        if rows[e]:
            _check_group(t, e, off[e], off[e + 1], act, out)


def test_bad_tables_are_skipped_and_reported():
    rows = [200, 300, 250, 274]
    t, off, desc, ws = _case(rows, 2592, 2464, C.SWIGLU, 9)
    n = sum(rows)
    bad = list(off)
    bad[4] = n + 5                      # the last group's range leaves the call's rows
    t["perm"][off[1] + 3] = n           # and one destination does
    out = _run(t, bad, desc, ws)
    assert C.ec2moe_last_device_error() == C.ERR_INVALID_ARG
    _check_group(t, 0, off[0], off[1], C.SWIGLU, out)
    _check_group(t, 2, off[2], off[3], C.SWIGLU, out)
    assert bool(out[t["perm"][off[3]:].long()].isnan().all())  # nothing written for the skipped group
    assert C.ec2moe_last_device_error() == C.OK


def test_zero_wait_budget_times_out_and_recovers():
    rows = [200, 300, 250, 274]
    t, off, desc, ws = _case(rows, 2592, 2464, C.SWIGLU, 11)
    old = C.ec2moe_get_wait_budget()
    try:
        C.ec2moe_set_wait_budget(0)
        _run(t, off, desc, ws)
        status = C.ec2moe_last_device_error()
    finally:
        C.ec2moe_set_wait_budget(old)
    assert status == C.ERR_TIMEOUT
    out = _run(t, off, desc, ws)
    assert C.ec2moe_last_device_error() == C.OK
    _check_group(t, 1, off[1], off[2], C.SWIGLU, out)
