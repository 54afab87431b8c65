"""Comparison helpers for the GPU parity tests (oracle vs the C-ABI path).

Tolerances (written in the tests that use them):
* routing indices and counts: bit-exact, except tokens whose oracle decision
  margin in log g is below ``TIE_GAP`` (near-ties; the kernel decides them in
  fp32); inside the top-k, slots whose adjacent margin is below ``TIE_GAP`` are
  compared as a set;
* combine weights: relative 2e-5 (fp32 logits of length d, fp32 exp/log);
* outputs: relative Frobenius error <= 1e-4 (fp32 layers) or 1e-2 (bf16
  layers, fp32 accumulation), max elementwise error <= 3e-2 for bf16.
"""

from __future__ import annotations

import numpy as np
import torch

from paper_2508_06024_gb300.synth import to_f64

TIE_GAP = 1e-6
W_RTOL = 2e-5


class LazyF64:
    """Per-expert float64 view of a stacked weight tensor, converted on access
    (keeps the oracle's memory at one expert for the large presets)."""

    def __init__(self, t: torch.Tensor):
        self.t = t
        self.shape = tuple(t.shape)

    def __getitem__(self, i):
        return to_f64(self.t[i])


def oracle_inputs(inp, lazy_experts: bool = False):
    out = {}
    for k, v in inp.items():
        if v is None:
            out[k] = None
        elif k == "mask":
            out[k] = v.to("cpu").numpy().astype(np.uint8)
        elif lazy_experts and k in ("W1", "W3", "W2", "W1s", "W3s", "W2s"):
            out[k] = LazyF64(v)
        else:
            out[k] = to_f64(v)
    return out


def routing_check(gpu_idx: np.ndarray, ref: dict, tie_gap: float = TIE_GAP):
    """Exact comparison of Top-k indices away from near-ties.

    Returns (n_compared, n_excluded).  Raises AssertionError on a mismatch."""
    oidx = ref["idx"]
    gb = ref["gap_boundary"]
    ga = ref["gap_adjacent"]
    T, k = oidx.shape
    assert gpu_idx.shape == (T, k)
    keep = gb >= tie_gap
    bad = []
    for t in np.nonzero(keep)[0]:
        a, b = gpu_idx[t].tolist(), oidx[t].tolist()
        if set(a) != set(b):
            bad.append(t)
            continue
        # runs of slots tied within tie_gap compare as sets
        start = 0
        for j in range(k):
            if j == k - 1 or ga[t, j] >= tie_gap:
                if set(a[start:j + 1]) != set(b[start:j + 1]):
                    bad.append(t)
                    break
                start = j + 1
    assert not bad, f"{len(bad)} tokens route differently, e.g. t={bad[:5]} gpu={gpu_idx[bad[0]]} ref={oidx[bad[0]]}"
    return int(keep.sum()), int((~keep).sum())


def weights_check(gpu_idx, gpu_w, ref, keep_mask, rtol=W_RTOL):
    """Combine weights of each selected expert, matched by expert id."""
    g = ref["g"] if "g" in ref else None
    w_ref = ref["w"]
    oidx = ref["idx"]
    for t in np.nonzero(keep_mask)[0]:
        ref_map = dict(zip(oidx[t].tolist(), w_ref[t].tolist()))
        for e, w in zip(gpu_idx[t].tolist(), gpu_w[t].tolist()):
            r = ref_map[e]
            assert abs(w - r) <= rtol * abs(r) + 1e-30, (t, e, w, r)
    return g


def rel_fro(a: np.ndarray, b: np.ndarray) -> float:
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def output_check(y_gpu: np.ndarray, y_ref: np.ndarray, bf16: bool, pair: bool = False):
    """The output tolerances against the oracle.  pair=True compares two GPU
    outputs that take different rounding paths: each lies within the bound of
    the exact result, so their difference is held to twice the max-abs bound
    (the Frobenius bound stays)."""
    err = rel_fro(y_gpu, y_ref)
    mx = float(np.abs(y_gpu - y_ref).max()) if y_ref.size else 0.0
    if bf16:
        mx_bound = 6e-2 if pair else 3e-2
        assert err <= 1e-2, f"relative Frobenius error {err:.3e} > 1e-2"
        assert mx <= mx_bound, f"max abs error {mx:.3e} > {mx_bound:.0e}"
    else:
        assert err <= 1e-4, f"relative Frobenius error {err:.3e} > 1e-4"
    return err, mx


def gemm_launches(call, name):
    """How many GEMM kernels called `name` the call launches; None where kernels
    cannot be traced (a process's first trace may come back empty)."""
    for _ in range(3):
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        names = [e.name for e in prof.events() if "gemm_kernel" in e.name]
        if names:
            return sum(name in n for n in names)
    return None
