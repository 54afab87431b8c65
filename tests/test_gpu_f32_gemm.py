"""The fp32 GEMM (three bf16 terms per operand) through the C ABI at the edges
of its tiles, against float64.

Bound per element: every product is exact up to 2^-24 |a b| (the three-term
split), a segment of 128 columns adds 8 MMAs of 16 products into one accumulator
and 40 into the other without rounding to nearest (at most 2^-23 of the running
magnitude per MMA; the second accumulator holds terms of 2^-8 |a b|), and the
K / 128 segments are added in fp32 (2^-24 each), so
|error| <= (8 + K / 64) 2^-23 sum_k |a_k b_k|.
"""

import pytest
import torch

from paper_2508_06024_gb300 import build as B
from paper_2508_06024_gb300 import ec2moe as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    C.load()


def _randn(seed, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda")


def _check(got, A, W, least=0.0):
    ref = A.double() @ W.double().T
    bound = least + (8 + A.shape[1] / 64) * 2.0 ** -23 * (A.double().abs() @ W.double().abs().T)
    assert bool(((got.double() - ref).abs() <= bound).all())


# rows around the 128-row tile, outputs around the 64- and 128-wide ones and at
# the smallest width, K below, at and past whole 64-column blocks
@pytest.mark.parametrize("T,d,r", [(1, 8, 8), (127, 72, 56), (128, 64, 64), (129, 520, 136), (300, 1024, 1160)])
def test_codec_f32_edges(T, d, r):
    X, Ve, Vd = _randn(1, T, d), _randn(2, r, d), _randn(3, d, r)
    desc = C.make_desc(T=T, d=d, E=8, d_ff=8, k=1, dtype=C.F32, r=r)
    Z = torch.full((T, r), float("nan"), device="cuda")
    Xh = torch.full((T, d), float("nan"), device="cuda")
    C.ec2moe_lr_encode(desc, X, Ve, Z)
    C.ec2moe_lr_decode(desc, Z, Vd, Xh)
    assert C.ec2moe_last_device_error() == C.OK
    _check(Z, X, Ve)
    _check(Xh, Z, Vd)


# K = 512 split over clusters of four as long as their tiles make one wave (36 fit
# at once, 38 are launched), of two beyond, and unsplit
@pytest.mark.parametrize("tiles", [36, 37, 38, 39, 76, 77, 153])
def test_f32_split_by_tile_count(tiles):
    T, d, r = tiles * 128 - 5, 512, 64
    X, Ve = _randn(1, T, d), _randn(2, r, d)
    desc = C.make_desc(T=T, d=d, E=8, d_ff=8, k=1, dtype=C.F32, r=r)
    Z = torch.full((T, r), float("nan"), device="cuda")
    C.ec2moe_lr_encode(desc, X, Ve, Z)
    assert C.ec2moe_last_device_error() == C.OK
    _check(Z, X, Ve)


def test_f32_rows_aligned_to_16_bytes_only():
    T, d, r = 150, 104, 72
    X = _randn(1, T * d + 4)[4:].view(T, d)  # 16-byte aligned, not 32
    Ve = _randn(2, r, d)
    desc = C.make_desc(T=T, d=d, E=8, d_ff=8, k=1, dtype=C.F32, r=r)
    Z = torch.empty(T, r, device="cuda")
    C.ec2moe_lr_encode(desc, X, Ve, Z)
    assert C.ec2moe_last_device_error() == C.OK
    _check(Z, X, Ve)


@pytest.mark.parametrize("act", [C.GELU, C.SWIGLU], ids=["gelu", "swiglu"])
@pytest.mark.parametrize("rows,d,ff", [([1, 0, 128, 130], 72, 40), ([0, 257, 0, 3], 200, 1096)],
                         ids=["narrow", "wide"])
def test_experts_f32_groups(rows, d, ff, act):
    E, n = len(rows), sum(rows)
    off = [sum(rows[:i]) for i in range(E + 1)]
    X, W1, W3, W2 = _randn(1, n, d), _randn(2, E, ff, d), _randn(3, E, ff, d), _randn(4, E, d, ff)
    perm = torch.randperm(n, generator=torch.Generator().manual_seed(5)).int().cuda()
    w = _randn(6, n).abs()
    desc = C.make_desc(T=n, d=d, E=E, d_ff=ff, k=1, act=act, dtype=C.F32)
    ws = torch.empty(C.ec2moe_experts_workspace_size(desc), dtype=torch.uint8, device="cuda")
    out = torch.full((n, d), float("nan"), device="cuda")
    C.ec2moe_experts(desc, X, torch.tensor(off, dtype=torch.int32, device="cuda"), W1, W3, W2, w, perm, out, ws,
                     ws.numel())
    assert C.ec2moe_last_device_error() == C.OK
    for e in range(E):
        if not rows[e]:
            continue
        x = X[off[e]:off[e + 1]].double()
        u = x @ W1[e].double().T
        h = torch.nn.functional.gelu(u) if act == C.GELU else torch.nn.functional.silu(u) * (x @ W3[e].double().T)
        p = perm[off[e]:off[e + 1]].long()
        ref = (h @ W2[e].double().T) * w[p].double()[:, None]
        err = float((out[p].double() - ref).norm() / ref.norm())
        assert err < 2e-6, err  # two chained fp32 products; a sequential FMA sum shows 1e-6


def test_f32_nonfinite_results_follow_the_fma_sum():
    X, V = _randn(1, 130, 128), _randn(2, 64, 128)
    X[3, 5] = float("inf")      # +-inf by the sign of the weight
    X[4, 7] = float("nan")
    X[129, 0] = 3.4e38          # rounds to infinity in bf16, finite in fp32
    V[:, 0] *= 0.5 / V[:, 0].abs().clamp(min=0.5)
    desc = C.make_desc(T=130, d=128, E=8, d_ff=8, k=1, dtype=C.F32, r=64)
    Z = torch.empty(130, 64, device="cuda")
    C.ec2moe_lr_encode(desc, X, V, Z)
    assert C.ec2moe_last_device_error() == C.OK
    assert torch.equal(Z[3], torch.sign(V[:, 5]) * float("inf"))
    assert bool(Z[4].isnan().all())
    keep = [i for i in range(130) if i not in (3, 4)]
    _check(Z[keep], X[keep], V)


def test_f32_recomputes_single_results():
    """One infinite weight in some of four neighbouring columns, which are
    computed again together: the finite ones keep their bits."""
    X, V = _randn(1, 130, 136), _randn(2, 72, 136)
    desc = C.make_desc(T=130, d=136, E=8, d_ff=8, k=1, dtype=C.F32, r=72)
    Z, ref = torch.empty(130, 72, device="cuda"), torch.empty(130, 72, device="cuda")
    C.ec2moe_lr_encode(desc, X, V, ref)
    bad = [1, 3, 40, 68, 69, 70, 71]
    V[bad, 135] = float("inf")
    C.ec2moe_lr_encode(desc, X, V, Z)
    assert C.ec2moe_last_device_error() == C.OK
    good = [i for i in range(72) if i not in bad]
    assert torch.equal(Z[:, good], ref[:, good])
    assert torch.equal(Z[:, bad], (torch.sign(X[:, 135:]) * float("inf")).expand(130, len(bad)))


# Operands over the whole exponent range: near and below the smallest normal
# number, products that small, and magnitudes whose scaled terms or sums
# overflow and are computed again.  Products and sums are exact down to far
# below fp32's smallest step, so the only absolute error is that of a result
# stored as a subnormal number (half of 2^-149).
@pytest.mark.parametrize("x2,w2", [(-120, 0), (0, -120), (-126, 10), (-140, 60), (-60, -60), (100, -100), (60, 30),
                                   (110, -60), (-70, 110)])
def test_f32_operand_range(x2, w2):
    T, d, r = 130, 200, 72
    X = (_randn(1, T, d).double() * 2.0 ** x2).float()
    V = (_randn(2, r, d).double() * 2.0 ** w2).float()
    desc = C.make_desc(T=T, d=d, E=8, d_ff=8, k=1, dtype=C.F32, r=r)
    Z = torch.empty(T, r, device="cuda")
    C.ec2moe_lr_encode(desc, X, V, Z)
    assert C.ec2moe_last_device_error() == C.OK
    _check(Z, X, V, 2.0 ** -149)


# Every kernel shape: 64- and 128-wide tiles, K split over a cluster and not,
# one tile and several per CTA.  With a budget of 0 a wait that is not satisfied
# at once gives up; the CTA still meets its cluster's barriers, ends its MMAs in
# flight and returns, and the next call finds nothing left over.
@pytest.mark.parametrize("T,d,r,decode", [(256, 512, 64, False), (4096, 768, 128, False), (300, 768, 128, True),
                                          (4096, 768, 128, True)],
                         ids=["64-wide-split", "128-wide-split", "64-wide", "128-wide"])
def test_f32_zero_wait_budget_times_out_and_recovers(T, d, r, decode):
    desc = C.make_desc(T=T, d=d, E=8, d_ff=8, k=1, dtype=C.F32, r=r)
    A, W = _randn(1, T, r if decode else d), _randn(2, *((d, r) if decode else (r, d)))
    call = C.ec2moe_lr_decode if decode else C.ec2moe_lr_encode
    ref, out = torch.empty(T, W.shape[0], device="cuda"), torch.empty(T, W.shape[0], device="cuda")
    call(desc, A, W, ref)
    assert C.ec2moe_last_device_error() == C.OK
    old = C.ec2moe_get_wait_budget()
    try:
        C.ec2moe_set_wait_budget(0)
        call(desc, A, W, out)
        status = C.ec2moe_last_device_error()
    finally:
        C.ec2moe_set_wait_budget(old)
    assert status == C.ERR_TIMEOUT
    assert C.ec2moe_last_device_error() == C.OK  # the error word was read and cleared
    call(desc, A, W, out)
    assert C.ec2moe_last_device_error() == C.OK
    assert torch.equal(out, ref)
