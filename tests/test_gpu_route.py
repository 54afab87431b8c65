"""Routing tables at the edges of the one-block kernel (a run of whole and
partial 32-entry pieces per warp, its largest size, the first size past it),
bit for bit against a stable sort; ids outside [0, E) are skipped."""

import numpy as np
import pytest
import torch

from paper_2508_06024_gb300 import build as B
from paper_2508_06024_gb300 import ec2moe as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    C.load()


@pytest.mark.parametrize("bad", [False, True], ids=["valid", "with-bad-ids"])
@pytest.mark.parametrize("n,E", [(1, 1), (31, 64), (1024, 128), (1025, 64), (12006, 64), (16384, 128), (16385, 33)])
def test_route_tables(n, E, bad):
    rng = np.random.default_rng(n + E)
    p = 1.0 / np.arange(1, E + 1)  # uneven load: runs of one expert within a warp
    idx = rng.choice(E, size=n, p=p / p.sum()).astype(np.int32)
    if bad:
        idx[rng.integers(0, n, size=max(1, n // 50))] = rng.choice([-1, E, 1 << 20])
    desc = C.make_desc(T=n, d=8, E=E, d_ff=8, k=1)
    out = {m: torch.full((s,), -7, dtype=torch.int32, device="cuda")
           for m, s in (("counts", E), ("offsets", E + 1), ("perm", n), ("inv", n))}
    ws = torch.empty(C.ec2moe_route_workspace_size(desc), dtype=torch.uint8, device="cuda")
    C.ec2moe_route(desc, torch.from_numpy(idx).cuda(), out["counts"], out["offsets"], out["perm"], out["inv"],
                   workspace=ws, ws_bytes=ws.numel())
    assert C.ec2moe_last_device_error() == (C.ERR_INVALID_ARG if bad else C.OK)
    ok = (idx >= 0) & (idx < E)
    counts = np.bincount(idx[ok], minlength=E)
    order = np.nonzero(ok)[0]
    order = order[np.argsort(idx[order], kind="stable")]
    inv = np.full(n, -1)
    inv[order] = np.arange(order.size)
    assert np.array_equal(out["counts"].cpu().numpy(), counts)
    assert np.array_equal(out["offsets"].cpu().numpy(), np.concatenate([[0], np.cumsum(counts)]))
    assert np.array_equal(out["perm"].cpu().numpy()[:order.size], order)
    assert np.array_equal(out["inv"].cpu().numpy(), inv)
