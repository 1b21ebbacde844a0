"""GPU parity of the multi-spike layer at the edges of its kernels' tiles
(two inputs per thread in the forward operand, sixteen samples per block in
the transposed one, 32 neurons per block of dC/dw^), from one to the largest
number of spikes and from 8 to 128 bins, against the float64 oracle. Bounds as
for the other multi-spike parity tests: times 1e-4 T_max, gradients 1e-3
relative L2 (fp32 arithmetic, three-product contractions).
"""

import numpy as np
import pytest

from helpers import grid_of, rel_l2
from oracle import multispike as oms
from test_gpu_multispike import compare_times, layer, lib, run  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,M", [((17, 9, 33, 8, 8), 8), ((1, 257, 31, 1, 2), 128), ((16, 31, 64, 5, 8), 33),
                                     ((33, 8, 1, 2, 1), 16), ((2, 1, 65, 8, 4), 64)])
def test_tile_edges(shape, M):
    B, N_in, N_out, F_in, F_out = shape
    tau_v, tau_I = 0.5, 0.25
    t, W, L = layer(11 + M, B, N_in, N_out, F_in, tau_v, tau_I, M=M)
    L["t_offset"] = 0.3 * 1.2 / M
    T, dt = grid_of(L)
    ctx = oms.dstd_forward_ms(t, W, T, dt, tau_v, tau_I, 1.0, F_out)
    ok = ctx["margin"] > 1e-4
    up = np.random.default_rng(M).normal(size=ctx["t"].shape)
    up = np.where(ok[..., None] & np.isfinite(ctx["t"]), up, 0.0)
    g = run(t, W, L, F_out, g_up=up.astype(np.float32))
    compare_times(g["t"], ctx, L)
    gW, gin, _ = oms.dstd_backward_ms(ctx, t, W, up.astype(np.float32).astype(np.float64), T, dt, tau_v, tau_I, 1.0)
    assert rel_l2(g["g_W"], gW) <= 1e-3
    assert rel_l2(g["g_in"], np.where(np.isfinite(t), gin, 0.0)) <= 1e-3
