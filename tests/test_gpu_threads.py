"""Several host threads, each with its own stream and buffers, calling layers of different sizes at the same time: no
call is refused, and every result is the one a single thread gets. A kernel's limit on dynamic shared memory is one
number for all threads, so a launch must not depend on the size another thread has just asked for."""

import math
import threading

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


def params(M):
    from paper_2607_14672_gb300 import dstd
    return dstd.params(dict(tau_v=INF, tau_I=INF, v_th=1.0, t_first=0.0, t_end=1.0, M=M, t_offset=0.0), 1.0)


def inputs(shape, w_shape, fan, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.rand(shape, device="cuda", generator=g)
    return t, 4.0 / fan + torch.randn(w_shape, device="cuda", generator=g) / math.sqrt(fan)


def dense(B, n_in, n_out, M, math_mode):
    from paper_2607_14672_gb300 import dstd
    t, W = inputs((B, n_in), (n_out, n_in), n_in, n_in)
    p = params(M)
    ws = torch.empty(dstd.dense_workspace_bytes(B, n_in, n_out, p, math_mode), dtype=torch.uint8, device="cuda")
    saved = torch.empty(dstd.dense_saved_bytes(B, n_out), dtype=torch.uint8, device="cuda")
    out = torch.empty(B, n_out, device="cuda")

    def call(stream):
        dstd.dense_fwd(t, W, p, math_mode, out, saved, None, ws, stream)
    return call, out


def exact(B, n_in, n_out):
    from paper_2607_14672_gb300 import dstd
    t, W = inputs((B, n_in), (n_out, n_in), n_in, n_in)
    p = params(16)
    ws = torch.empty(dstd.exact_workspace_bytes(B, n_in, n_out), dtype=torch.uint8, device="cuda")
    out = torch.empty(B, n_out, device="cuda")

    def call(stream):
        dstd.exact_fwd(t, W, p, out, ws, stream)
    return call, out


def conv(B, H, C, O, M):
    from paper_2607_14672_gb300 import dstd
    t, W = inputs((B, H, H, C), (O, 3, 3, C), 9 * C, H)
    p = params(M)
    ws = torch.empty(dstd.conv_workspace_bytes(B, H, H, C, O, 3, 1, 1, p, "bf16"), dtype=torch.uint8, device="cuda")
    saved = torch.empty(dstd.dense_saved_bytes(B * H * H, O), dtype=torch.uint8, device="cuda")
    out, up = torch.empty(B, H, H, O, device="cuda"), torch.ones(B, H, H, O, device="cuda")
    g_in, g_W = torch.empty_like(t), torch.empty_like(W)

    def call(stream):
        dstd.conv_fwd(t, W, 1, 1, p, "bf16", out, saved, None, ws, stream)
        dstd.conv_bwd(t, W, out, saved, up, 1, 1, p, "bf16", g_in, g_W, ws, stream)
    return call, out


CASES = {
    "few_outputs": lambda: [dense(8, 784, 10, 32, "f32"), dense(8, 64, 12, 32, "f32")],
    "exact": lambda: [exact(2, 8000, 8), exact(2, 4000, 8)],
    "conv_128": lambda: [conv(2, 8, 128, 128, 64), conv(2, 8, 128, 128, 32)],
    "conv_64": lambda: [conv(4, 2, 64, 64, 64), conv(4, 2, 64, 64, 32), conv(2, 14, 64, 64, 32)],
}


@pytest.mark.parametrize("name", CASES)
def test_threads_do_not_refuse_each_other(name):
    work = CASES[name]()
    torch.cuda.synchronize()
    want = []
    for call, out in work:
        call(torch.cuda.current_stream())
        torch.cuda.synchronize()
        want.append(out.clone())
    errors, start = [], threading.Barrier(len(work))

    def loop(call):
        stream = torch.cuda.Stream()
        start.wait()
        try:
            for i in range(600):
                call(stream)
                if i % 50 == 49:
                    stream.synchronize()
        except Exception as e:
            errors.append(repr(e))
        stream.synchronize()

    threads = [threading.Thread(target=loop, args=(c,)) for c, _ in work]
    for x in threads:
        x.start()
    for x in threads:
        x.join()
    assert errors == []
    for (_, out), w in zip(work, want):
        assert torch.equal(out, w)
