"""The conv contractions that take each source row (dW: each column) once (the default path) against the one-row-at-a-time kernels
(operand policy 2, whose results the conv parity tests hold to the oracle).

Forward: the same products in the same order per output, so spike times and saved state are equal bit for bit.
Input-time gradient: the same products in the same order too; the two bins of an input may be added in either order.
Weight gradient: fp32 sums in another order, at most a few hundred accumulations of 2^-24 each: 2e-5 relative L2.
Shapes: widths that the position tile does not divide, odd grids at stride 2, one image row, 1x1, 5x5 and 7x7
filters, filters resident and streamed, several channel blocks, padded input channels, chunks."""

import math

import pytest
import torch

pytestmark = pytest.mark.gpu

INF = math.inf


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2607_14672_gb300 import build, dstd
    build.build()
    dstd.load()
    assert dstd.device_status(clear=True) == 0
    yield
    assert dstd.device_status(clear=True) == 0


def run(B, H, Wd, C, O, k, stride, pad, M, tau, policy, chunk=0):
    from paper_2607_14672_gb300 import dstd
    g = torch.Generator(device="cuda")
    g.manual_seed(H * 1000 + C + O + k)
    t = torch.rand((B, H, Wd, C), device="cuda", generator=g)
    t[torch.rand(t.shape, device="cuda", generator=g) < 0.3] = INF
    fan = C * k * k
    mean = {(INF, INF): 4.0, (0.4, 0.2): 28.0}.get(tau, 16.0)
    W = mean / fan + torch.randn((O, k, k, C), device="cuda", generator=g) / math.sqrt(fan)
    L = dict(tau_v=tau[0], tau_I=tau[1], v_th=1.0, t_first=-0.03, t_end=1.1, M=M, t_offset=0.2 * 1.13 / M, t_head_l=0.3,
             t_tail_l=0.8, gamma_head=0.05, gamma_tail=0.01, gamma_q=1e-3)
    Ho, Wo = dstd.conv_out_hw(H, Wd, k, stride, pad)
    p = dstd.params(L, 1.0 / (B * Ho * Wo))
    up = 1e-2 * torch.randn((B, Ho, Wo, O), device="cuda", generator=g)
    prev, pc = dstd.conv_set_operand_policy(policy), dstd.conv_set_chunk_images(chunk)
    try:
        ws = torch.full((dstd.conv_workspace_bytes(B, H, Wd, C, O, k, stride, pad, p, "bf16"),), 0xFF,
                        dtype=torch.uint8, device="cuda")
        out = torch.full((B, Ho, Wo, O), -7.0, device="cuda")
        saved = torch.zeros(dstd.dense_saved_bytes(B * Ho * Wo, O), dtype=torch.uint8, device="cuda")
        pen = torch.zeros(4, device="cuda")
        g_in, g_W = torch.full_like(t, 7.0), torch.full_like(W, 7.0)
        dstd.conv_fwd(t, W, stride, pad, p, "bf16", out, saved, pen, ws)
        dstd.conv_bwd(t, W, out, saved, up, stride, pad, p, "bf16", g_in, g_W, ws)
        torch.cuda.synchronize()
        assert dstd.device_status(clear=True) == 0
    finally:
        dstd.conv_set_operand_policy(prev)
        dstd.conv_set_chunk_images(pc)
    return out, saved, pen, g_in, g_W


def rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm().clamp(min=1e-30))


# H, W, C_in, C_out, k, stride, pad, M, tau; the batch is taken just large enough for the row kernels to be chosen
CASES = [
    (28, 28, 64, 64, 3, 1, 1, 64, (1.0, 0.25)),
    (7, 7, 64, 64, 3, 1, 1, 50, (0.5, 0.25)),        # odd width, M below the padded 64
    (5, 9, 64, 64, 3, 1, 1, 20, (INF, INF)),         # rows and columns differ, four positions per tile
    (1, 6, 64, 64, 3, 1, 1, 32, (INF, INF)),         # one image row
    (6, 6, 3, 64, 3, 1, 1, 32, (INF, INF)),          # padded input channels
    (9, 9, 64, 128, 3, 2, 1, 64, (1.0, 0.25)),       # stride 2 on an odd grid, two channel blocks in dS
    (8, 8, 64, 128, 3, 2, 1, 33, (0.4, 0.2)),        # and on an even one
    (10, 10, 64, 64, 3, 2, 1, 32, (INF, INF)),       # stride 2, one channel block
    (14, 14, 64, 128, 3, 1, 1, 64, (1.0, 0.25)),     # two channel blocks in dS
    (7, 7, 64, 256, 3, 1, 1, 32, (0.5, 0.25)),       # four, at a width that the tile does not divide
    (8, 8, 64, 64, 5, 1, 2, 20, (INF, INF)),         # 5x5
    (8, 8, 64, 64, 1, 1, 0, 32, (INF, INF)),         # 1x1
    (9, 9, 64, 64, 7, 1, 3, 32, (0.5, 0.25)),        # 7x7
    (9, 9, 64, 64, 5, 2, 2, 64, (0.5, 0.25)),        # 5x5 at stride 2
    (8, 8, 64, 64, 3, 1, 0, 32, (INF, INF)),         # no padding
    (8, 8, 64, 64, 3, 1, 2, 32, (INF, INF)),         # padding k - 1
]


def batch(case):
    Ho, Wo = ((case[i] + 2 * case[6] - case[4]) // case[5] + 1 for i in (0, 1))
    # forward: 300 output positions per SM; dS alone (more than 64 output channels or stride 2): 20 input positions
    need = 300 * 152 // (Ho * Wo) if case[3] == 64 and case[5] == 1 else 20 * 152 // (case[0] * case[1])
    return need + 1


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c[:8]))
def test_rows_match_one_row_at_a_time(case):
    B = batch(case)
    a, b = run(B, *case, policy=0), run(B, *case, policy=2)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert torch.isfinite(a[0]).any()
    assert rel(a[2], b[2]) <= 1e-5
    assert rel(a[3], b[3]) <= 2e-5
    assert rel(a[4], b[4]) <= 2e-5


@pytest.mark.parametrize("case", [(3, 14, 14, 128, 128, 3, 1, 1, 64, (1.0, 0.25)), (2, 7, 9, 64, 256, 3, 1, 1, 50, (0.5, 0.25)),
                                  (1, 1, 1, 64, 64, 3, 1, 1, 32, (INF, INF)), (5, 4, 3, 192, 64, 3, 1, 1, 20, (INF, INF)),
                                  (2, 6, 5, 5, 64, 3, 1, 0, 64, (0.5, 0.25)), (700, 3, 3, 64, 128, 3, 1, 2, 40, (0.4, 0.2))],
                         ids=lambda c: "-".join(str(x) for x in c[:9]))
def test_weight_gradient_by_columns(case):
    """dW of 3x3 layers at stride 1: both tile widths, several channel blocks and column tiles, padded channels, rows
    split over few and many CTAs, a single position."""
    a, b = run(*case, policy=0), run(*case, policy=2)
    assert torch.equal(a[0], b[0]) and (b[4] != 0).any()
    assert rel(a[4], b[4]) <= 2e-5


def test_rows_chunks_agree():
    case = (6, 6, 64, 64, 3, 1, 1, 32, (INF, INF))
    B = batch(case)
    a, b = run(2 * B, *case, policy=0), run(2 * B, *case, policy=0, chunk=B)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(a[3], b[3])
    assert rel(a[4], b[4]) <= 2e-5
