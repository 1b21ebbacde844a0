"""The dense contraction's kernels against each other and the oracle. Order of the output tiles: bands of 12 row tiles (128 rows each) on single CTAs, of 6
(256 rows) on SM pairs. Shapes whose last band is partial, in both operand modes and on both kernels, against the
oracle's w^ within the bound of the contraction's own parity test."""

import numpy as np
import pytest
import torch

from helpers import bf16, dense_layer, f32
from oracle import dstd as odstd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2607_14672_gb300 import build, dstd
    build.build()
    dstd.load()
    assert dstd.device_status(clear=True) == 0
    yield
    assert dstd.device_status(clear=True) == 0


@pytest.mark.parametrize("math_mode", ["x3", "bf16"])
@pytest.mark.parametrize("policy", [1, 2], ids=["pairs", "single"])
@pytest.mark.parametrize("B,N_in,N_out", [(64, 72, 1700), (52, 40, 1541)])   # 14 and 13 row tiles; 8 and 7 pair rows
def test_partial_band(math_mode, policy, B, N_in, N_out):
    from paper_2607_14672_gb300 import dstd
    M = 32
    t_in, layer = dense_layer(B, N_in, N_out, M, 0.5, 0.25, seed=N_in, t_offset=0.01)
    t_in, W = f32(t_in), f32(layer["W"])
    p = dstd.params(layer, 1.0 / B)
    dev = lambda x: torch.tensor(x, dtype=torch.float32, device="cuda").contiguous()
    ws = torch.empty(dstd.dense_workspace_bytes(B, N_in, N_out, p, math_mode), dtype=torch.uint8, device="cuda")
    what = torch.empty(B, N_out, M, device="cuda")
    prev = dstd.set_pair_policy(policy)
    try:
        dstd.dense_what(dev(t_in), dev(W), p, math_mode, what, ws)
        torch.cuda.synchronize()
    finally:
        dstd.set_pair_policy(prev)
    T, dt = odstd.grid(layer["t_first"], layer["t_end"], M, layer["t_offset"])
    s = odstd.binning(t_in, T, dt, 0.5, 0.25)
    ds = odstd.binning(t_in, T, dt, 0.5, 0.25, derivative=True)
    prod = lambda a, b: np.matmul(a.reshape(B * M, N_in), b.T).reshape(B, M, N_out).transpose(0, 2, 1)
    aW = np.abs(W)
    bound = 3e-7 * prod(np.abs(ds), aW) + 1e-7          # spike times known to about 1e-7
    if math_mode == "bf16":
        ref = prod(bf16(s), bf16(W))
        # one bf16 step in single terms (at most the largest product) and the fp32 accumulation
        bound = bound + 2.0 ** -14 * prod(np.abs(s), aW) + 2.0 ** -8 * np.abs(s).max() * aW.max()
    else:
        ref = prod(s, W)
        bound = bound + 3e-5 * prod(np.abs(s), aW)
    err = np.abs(what.cpu().numpy().astype(np.float64) - ref)
    assert (err <= bound).all(), float(np.max(err / bound))


@pytest.mark.parametrize("B,N_in,N_out,M", [(9, 300, 140, 8), (5, 257, 70, 16), (4, 520, 200, 20), (3, 200, 300, 50),
                                            (2, 513, 333, 100), (64, 1700, 72, 32), (1, 8, 129, 128)])
def test_input_gradient_on_pairs(B, N_in, N_out, M):
    """bf16 dS with the input-time gradient in its epilogue: SM pairs and single CTAs add in the same order per
    accumulator, so the gradient is equal bit for bit (every padded grid size, ragged rows and columns)."""
    from paper_2607_14672_gb300 import dstd
    t_in, layer = dense_layer(B, N_in, N_out, M, 0.5, 0.25, seed=N_in + M, t_offset=0.001, fire=0.6)
    p = dstd.params(layer, 1.0 / B)
    dev = lambda x: torch.tensor(np.asarray(x), dtype=torch.float32, device="cuda").contiguous()
    t, W = dev(t_in), dev(layer["W"])
    up = dev(np.random.default_rng(M).normal(size=(B, N_out)))
    ws = torch.empty(dstd.dense_workspace_bytes(B, N_in, N_out, p, "bf16"), dtype=torch.uint8, device="cuda")
    out = torch.empty(B, N_out, device="cuda")
    saved = torch.empty(dstd.dense_saved_bytes(B, N_out), dtype=torch.uint8, device="cuda")
    dstd.dense_fwd(t, W, p, "bf16", out, saved, torch.empty(4, device="cuda"), ws)
    got = []
    for policy in (1, 2):
        g_in, g_W = torch.full_like(t, 7.0), torch.empty_like(W)
        prev = dstd.set_pair_policy(policy)
        try:
            dstd.dense_bwd(t, W, out, saved, up, p, "bf16", g_in, g_W, ws)
            torch.cuda.synchronize()
        finally:
            dstd.set_pair_policy(prev)
        got.append(g_in)
    assert torch.isfinite(out).any() and (got[0] != 0).any()
    assert torch.equal(got[0], got[1])
