"""The benchmark's work per kernel kind follows the kernels that the library takes: no bytes of a w^ that the fused
forward never writes, and 8-byte records where the operand is generated on chip."""

import os
import shutil
from types import SimpleNamespace

import pytest

B, M = 256, 64


def net(*layers):
    """layers: (H, C_in, C_out, stride) of 3x3 conv layers."""
    from paper_2607_14672_gb300 import dstd
    L = dict(tau_v=1.0, tau_I=0.25, v_th=1.0, t_first=0.0, t_end=1.2, M=M, t_offset=0.0)
    p = dstd.params(L, 1.0)
    return SimpleNamespace(B=B, math="bf16", layers=[L] * len(layers), p=[p] * len(layers),
                           W=[SimpleNamespace(shape=(O, 3, 3, C)) for _, C, O, _ in layers],
                           geom=[(H, H, C, 3, st, 1) for H, C, _, st in layers])


@pytest.fixture(scope="module")
def units():
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    from paper_2607_14672_gb300 import build, dstd
    build.build()
    dstd.load()
    from bench import conv_step_units
    return conv_step_units


def test_fused_layers_have_no_scan_bytes(units):
    _, _, b = units(net((28, 64, 64, 1), (28, 64, 128, 2), (14, 128, 128, 1)))
    assert "scan_solve" not in b
    from paper_2607_14672_gb300 import dstd
    prev = dstd.conv_set_operand_policy(1)               # operand generated, scan in a kernel of its own
    try:
        _, _, b = units(net((14, 128, 128, 1)))
    finally:
        dstd.conv_set_operand_policy(prev)
    n = B * 14 * 14 * 128
    assert b["scan_solve"] == n * (M * 4 + 16) and b["binning"] == b["binning_T"] == n * 12


def test_binning_bytes_follow_the_route(units):
    rows = B * 28 * 28 * 64
    _, _, b = units(net((28, 64, 64, 1)))
    assert b["binning"] == b["binning_T"] == rows * 12
    _, _, b = units(net((28, 64, 128, 2)))
    assert b["binning"] == b["binning_T"] == rows * (4 + 2 * M)
    n = net((2, 64, 64, 1))                              # small: S in both directions
    _, _, b = units(n)
    assert b["binning"] == b["binning_T"] == B * 4 * 64 * (4 + 2 * M)
