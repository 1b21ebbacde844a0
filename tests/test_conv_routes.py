"""Which kernels a conv layer takes (dstd_conv_route): the rules on the host, and, on the GPU, that the shapes meant
to check the kernels by source rows against the one-row-at-a-time kernels do take them.

Forward by rows: 64 output channels, one block of 64 input channels (or fewer, padded), stride 1, filters above 1x1
that come at least a filter row at a time, 300 output positions per SM. dS by rows: one block of input channels, 20
input positions per SM, at most eight output rows in flight (four at stride 2). Both only where they are the faster
kernels, as the measured times say. Forward results are equal bit for bit, input-time gradients to 1e-5 relative L2
(the two bins of an input may be added in either order), as in test_gpu_conv_rows.py.

dW by columns: 3x3 at stride 1, 64 output channels, or a multiple of 128 with 64 grid steps, on the side of the
measured crossing where it is the faster one. Weight gradients are fp32 sums in another order: 2e-5 relative L2, as in
test_gpu_conv_rows.py."""

import math
import os
import shutil

import pytest

INF = math.inf

# H, W, C_in, C_out, k, stride, pad, M, tau, and the kernels by rows that a large batch takes
LARGE = [
    (28, 28, 64, 64, 3, 1, 1, 64, (1.0, 0.25), {"fwd_rows", "ds_rows"}),
    (7, 7, 64, 64, 3, 1, 1, 50, (0.5, 0.25), {"fwd_rows", "ds_rows"}),
    (1, 6, 64, 64, 3, 1, 1, 32, (INF, INF), {"fwd_rows", "ds_rows"}),
    (6, 6, 3, 64, 3, 1, 1, 32, (INF, INF), {"fwd_rows", "ds_rows"}),
    (8, 8, 64, 64, 2, 1, 1, 32, (INF, INF), {"fwd_rows", "ds_rows"}),
    (9, 9, 64, 64, 4, 1, 2, 32, (INF, INF), {"fwd_rows", "ds_rows"}),     # filters a row at a time
    (7, 7, 64, 64, 5, 1, 2, 20, (INF, INF), {"fwd_rows", "ds_rows"}),
    (7, 7, 64, 64, 3, 1, 1, 64, (INF, INF), {"fwd_rows", "ds_rows"}),
    (28, 28, 64, 64, 3, 1, 1, 32, (INF, INF), {"fwd_rows", "ds_rows"}),
    (28, 28, 64, 64, 3, 1, 1, 64, (INF, INF), {"ds_rows"}),              # a light scan beside row boxes
    (4, 4, 64, 64, 3, 1, 1, 32, (0.5, 0.25), {"fwd_rows"}),              # dS tiles twice as wide as the image
    (9, 9, 64, 64, 7, 1, 3, 32, (0.5, 0.25), {"ds_rows"}),               # filters a column at a time: no forward
    (7, 7, 64, 64, 5, 1, 2, 64, (0.5, 0.25), {"ds_rows"}),
    (8, 8, 64, 64, 1, 1, 0, 32, (INF, INF), {"ds_rows"}),
    (9, 9, 64, 128, 3, 2, 1, 64, (1.0, 0.25), {"ds_rows"}),
    (10, 10, 64, 64, 3, 2, 1, 32, (INF, INF), {"ds_rows"}),
    (7, 9, 64, 128, 3, 1, 1, 64, (0.5, 0.25), {"ds_rows"}),
    (7, 7, 64, 128, 3, 1, 1, 32, (0.5, 0.25), {"ds_rows"}),
    (4, 4, 64, 128, 3, 1, 1, 64, (0.5, 0.25), {"ds_rows"}),
    (8, 8, 64, 256, 3, 1, 1, 32, (0.5, 0.25), {"ds_rows"}),
    (3, 3, 64, 256, 1, 1, 0, 32, (0.5, 0.25), {"ds_rows"}),
    (4, 4, 64, 512, 5, 1, 2, 64, (0.5, 0.25), {"ds_rows"}),
    (7, 7, 64, 256, 3, 1, 1, 32, (0.5, 0.25), set()),                    # four channel blocks in one stage: too large
    (9, 9, 64, 64, 5, 2, 2, 64, (0.5, 0.25), set()),     # six output rows in flight, four accumulators
    (28, 28, 64, 128, 3, 1, 1, 32, (1.0, 0.25), set()),  # from here on: 0.6 to 0.9 of the other kernels' speed
    (28, 28, 64, 64, 5, 1, 2, 20, (INF, INF), set()),    # (those have row boxes)
    (28, 28, 64, 64, 5, 1, 2, 64, (1.0, 0.25), set()),
    (28, 28, 64, 64, 7, 1, 3, 64, (1.0, 0.25), set()),
    (14, 14, 128, 128, 3, 1, 1, 64, (1.0, 0.25), set()),
    (14, 14, 128, 64, 3, 1, 1, 64, (1.0, 0.25), set()),
]
ROWS = {"fwd_rows", "ds_rows"}

# B, H, W, C_in, C_out, pad, M of 3x3 layers at stride 1: clearly faster by columns ...
COLUMNS = [
    (256, 28, 28, 64, 64, 1, 64), (256, 28, 28, 3, 64, 1, 64), (82, 14, 14, 64, 64, 1, 64), (82, 7, 7, 256, 64, 1, 64),
    (256, 14, 14, 128, 128, 1, 64), (164, 14, 14, 256, 256, 1, 64),
    (12, 2, 2, 64, 64, 1, 32), (25, 1, 1, 64, 64, 1, 32), (12, 2, 2, 64, 64, 1, 64),
    (3, 4, 3, 192, 64, 1, 20), (2, 6, 5, 5, 64, 0, 32), (12, 2, 2, 128, 128, 1, 64), (25, 1, 1, 128, 128, 1, 64),
    (2, 3, 4, 64, 128, 1, 50), (3, 2, 2, 128, 256, 2, 33), (800, 5, 4, 64, 64, 2, 40), (700, 9, 9, 64, 128, 0, 64),
    (347, 11, 11, 64, 64, 1, 32), (195, 16, 16, 64, 64, 1, 32), (92, 24, 24, 64, 64, 1, 32),
]
# ... and clearly slower
TAPS = [
    (250, 2, 2, 64, 64, 1, 64), (1, 28, 28, 64, 64, 1, 64), (1, 28, 28, 128, 64, 1, 64), (111, 3, 3, 64, 64, 1, 64),
    (40, 10, 10, 128, 64, 1, 32), (40, 10, 10, 256, 64, 1, 32), (50, 2, 2, 256, 256, 1, 64), (12, 2, 2, 512, 512, 1, 64),
    (62, 4, 4, 512, 512, 1, 64), (20, 14, 14, 128, 128, 1, 64), (1000, 2, 2, 128, 128, 1, 64),
    (256, 14, 14, 128, 128, 1, 32),
]


@pytest.fixture(scope="module")
def lib():
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    from paper_2607_14672_gb300 import build, dstd
    build.build()
    return dstd.load()


def params(M, tau):
    from paper_2607_14672_gb300 import dstd
    return dstd.params(dict(tau_v=tau[0], tau_I=tau[1], v_th=1.0, t_first=-0.03, t_end=1.1, M=M,
                            t_offset=0.2 * 1.13 / M), 1.0)


def route(B, case, policy=0, math_mode="bf16"):
    from paper_2607_14672_gb300 import dstd
    prev = dstd.conv_set_operand_policy(policy)
    try:
        return dstd.conv_route(B, *case[:7], params(case[7], case[8]), math_mode)
    finally:
        dstd.conv_set_operand_policy(prev)


@pytest.mark.parametrize("case", LARGE, ids=lambda c: "-".join(str(x) for x in c[:8]))
def test_rules(lib, case):
    B = 400 * 200 // (case[0] * case[1]) + 1             # above the bounds on up to 200 SMs
    assert route(B, case) & ROWS == case[9]
    assert route(1, case) & ROWS == set() or case[0] * case[1] >= 20 * 148
    for policy in (1, 2):
        r = route(B, case, policy)
        assert r & (ROWS | {"dw_columns"}) == set()
        assert ("fwd_binned" in r, "dw_binned" in r) == ((policy == 2 or case[2] < 64,) * 2)
        assert ("fused_scan" in r) == ("fwd_binned" in r)
    r = route(B, case)
    assert {"implicit", "fused_scan"} <= r and ("fwd_binned" in r) != ("fwd_rows" in r)
    assert route(B, case, math_mode="x3") == set()       # the im2col path


def test_refused_and_other_paths(lib):
    from paper_2607_14672_gb300 import dstd
    p = params(32, (0.5, 0.25))
    assert dstd.conv_route(4, 8, 8, 100, 64, 3, 1, 1, p, "bf16") == set()   # neither below 64 channels nor a multiple
    for bad, code in (((4, 8, 8, 64, 64, 3, 1, 3, p, "bf16"), -1), ((0, 8, 8, 64, 64, 3, 1, 1, p, "bf16"), -1),
                      ((4, 8, 8, 64, 64, 3, 1, 1, p, "f32"), -2),
                      ((4, 8, 8, 64, 64, 3, 1, 1, params(200, (0.5, 0.25)), "bf16"), -2)):
        with pytest.raises(dstd.DstdError) as e:
            dstd.conv_route(*bad)
        assert e.value.code == code


def dw_case(c):
    B, H, W, C, O, pad, M = c
    return H, W, C, O, 3, 1, pad, M, (1.0, 0.25) if M > 32 else (INF, INF)


@pytest.mark.parametrize("c", COLUMNS + TAPS, ids=lambda c: "-".join(str(x) for x in c))
def test_columns_where_they_are_faster(lib, c):
    r = route(c[0], dw_case(c))
    assert ("dw_columns" in r) == (c in COLUMNS)
    assert ("dw_binned" in r) == (c not in COLUMNS or c[4] != 64)
    assert "dw_columns" not in route(c[0], dw_case(c), policy=2)


@pytest.mark.gpu
@pytest.mark.parametrize("c", [c for c in COLUMNS if c[0] * c[1] * c[2] < 60000], ids=lambda c: "-".join(str(x) for x in c))
def test_columns_are_taken_and_match(lib, c):
    import torch
    from paper_2607_14672_gb300 import dstd
    from test_gpu_conv_rows import rel, run
    dstd.device_status(clear=True)
    case = dw_case(c)
    assert "dw_columns" in route(c[0], case) and "dw_columns" not in route(c[0], case, policy=2)
    a, b = run(c[0], *case, policy=0), run(c[0], *case, policy=2)
    assert torch.equal(a[0], b[0]) and (b[4] != 0).any()
    assert rel(a[4], b[4]) <= 2e-5


@pytest.mark.gpu
@pytest.mark.parametrize("case", [c for c in LARGE if c[9]], ids=lambda c: "-".join(str(x) for x in c[:8]))
def test_rows_are_taken_and_match(lib, case):
    import torch
    from paper_2607_14672_gb300 import dstd
    from test_gpu_conv_rows import rel, run
    dstd.device_status(clear=True)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    Ho, Wo = dstd.conv_out_hw(case[0], case[1], *case[4:7])
    B = (300 * sms // (Ho * Wo) if "fwd_rows" in case[9] else 60 * sms // (case[0] * case[1])) + 1
    assert route(B, case) & ROWS == case[9] and route(B, case, policy=2) & ROWS == set()
    a, b = run(B, *case[:9], policy=0), run(B, *case[:9], policy=2)
    assert torch.isfinite(a[0]).any() and (a[3] != 0).any()
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert rel(a[3], b[3]) <= 1e-5
