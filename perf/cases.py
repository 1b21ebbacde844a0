"""Performance cases of the DSTD layers and networks, through the public entry points.

Sizes are those of this package's own configurations (``configs.py``): the
single 64 -> 32 layer, the 784-800-800-10 MLP, the N -> N layers, the layer
shapes of the conv networks and the multi-spike layer, with batch sizes from
a handful of samples to the training batches. ``draw`` spreads layers over
the same ranges, odd sizes included. ``exact`` restates every layer in 64
bits with plain torch: for the bf16 mode on operands rounded to bf16, which
is what that mode computes with.

A single layer takes part in training (``bwd`` true): forward, then backward
with an upstream gradient, the input-time gradient and the weight gradient.
With ``bwd`` false it is inference. Networks run through ``net.py``.
"""

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2607_14672_gb300 import configs, dstd, net

INF = math.inf
GRAD_SCALE = 1e-2          # upstream gradient, about a mini-batch mean's

# mean weight x fan-in at which most neurons of a layer fire, per (tau_m, tau_s): dense layers with
# inputs spread over the window, conv layers with inputs that are the previous layer's spikes
DENSE_MEAN = {"0.5,0.25": 16.0, "0.4,0.2": 17.4, "1.0,0.25": 12.0, "inf,inf": 4.0}
CONV_MEAN = {"0.5,0.25": 14.0, "0.4,0.2": 17.0, "1.0,0.25": 12.0, "inf,inf": 4.0}


def _dense(name, B, n_in, n_out, M, math_mode, tau, bwd=True):
    return dict(name=name, kind="dense", B=B, n_in=n_in, n_out=n_out, M=M, math=math_mode, tau=tau, bwd=bwd)


def _conv(name, B, H, c_in, c_out, k, stride, M, math_mode, tau, bwd=True):
    return dict(name=name, kind="conv", B=B, H=H, c_in=c_in, c_out=c_out, k=k, stride=stride, M=M, math=math_mode,
                tau=tau, bwd=bwd)


def listed():
    return [
        # one small fp32 layer in training (config 1): launches and latency only
        _dense("layer_64_32_f32", 8, 64, 32, 16, "f32", "0.5,0.25"),
        # answering a few requests at a time with the 784-800-800-10 MLP: latency
        dict(name="mlp_infer_b4", kind="mlp", B=4, M=32, bwd=False),
        # the MLP's training pass (config 2): forward, cross-entropy, backward
        dict(name="mlp_train_b256", kind="mlp", B=256, M=32, bwd=True),
        # a wide fp32-accurate layer in training (config 3, N = 4096)
        _dense("dense_4096_x3", 128, 4096, 4096, 32, "x3", "0.4,0.2"),
        # the widest layer on the finest grid (config 3, N = 16384, M = 128), bf16 operands
        _dense("dense_16384_bf16", 128, 16384, 16384, 128, "bf16", "0.4,0.2"),
        # conv layers in training at the 20-layer network's batch (config 5: layers 2-6, 7, 8-13)
        _conv("conv_64_28", 256, 28, 64, 64, 3, 1, 64, "bf16", "1.0,0.25"),
        _conv("conv_64_128_s2", 256, 28, 64, 128, 3, 2, 64, "bf16", "1.0,0.25"),
        _conv("conv_128_14", 256, 14, 128, 128, 3, 1, 64, "bf16", "1.0,0.25"),
        # the last conv layer of the 9-layer network (config 4): few positions, many channels
        _conv("conv_512_4", 128, 4, 512, 512, 3, 1, 32, "bf16", "inf,inf"),
        # the 5x5 layer of Syn-SNN-9: a grid that is no power of two, a batch of 50
        _conv("conv_5x5_m20", 50, 8, 128, 128, 5, 1, 20, "bf16", "inf,inf"),
        # inference of the whole 20-layer skip-and-delay network (Syn-SNN-20)
        dict(name="syn20_infer_b50", kind="syn20", B=50, M=20, bwd=False),
        # a multi-spike layer in training
        dict(name="multispike_800", kind="ms", B=256, n_in=800, n_out=800, M=32, spikes=4, math="x3",
             tau="0.5,0.25", bwd=True),
    ]


# -- drawn cases ------------------------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _conv_cost(c):
    pad_in = 64 * -(-c["c_in"] // 64)
    pad_out = 64 * -(-c["c_out"] // 64)
    Mp = max(8, 1 << (c["M"] - 1).bit_length())
    return c["B"] * (c["H"] / c["stride"]) ** 2 * Mp * c["k"] ** 2 * pad_in * pad_out * (3 if c["math"] == "x3" else 1)


def draw(rng):
    kind = rng.choice(["dense", "dense", "dense", "conv", "conv", "conv", "mlp", "ms"])
    bwd = rng.random() < 0.7
    tau = rng.choice(["0.5,0.25", "0.4,0.2", "1.0,0.25", "inf,inf"])
    if kind == "mlp":
        return dict(kind="mlp", B=_log_int(rng, 1, 512), M=rng.choice([8, 16, 20, 32, 48, 64]), bwd=bwd)
    if kind == "ms":
        n = [_log_int(rng, 32, 2048) for _ in range(2)]
        return dict(kind="ms", B=_log_int(rng, 4, 256), n_in=n[0], n_out=n[1], M=rng.choice([12, 16, 20, 32]),
                    spikes=rng.randint(2, 5), math="x3", tau="0.5,0.25", bwd=bwd)
    if kind == "dense":
        while True:
            n = [_log_int(rng, 32, 16384) for _ in range(2)]
            if rng.random() < 0.4:
                n = [8 * -(-v // 8) for v in n]
            c = dict(kind="dense", B=_log_int(rng, 1, 512), n_in=n[0], n_out=n[1],
                     M=rng.choice([8, 16, 20, 32, 50, 64, 100, 128]),
                     math=rng.choice(["x3", "x3", "x3", "bf16", "bf16", "f32"]), tau=tau, bwd=bwd)
            cost = c["B"] * c["M"] * n[0] * n[1] * {"x3": 3, "bf16": 1, "f32": 40}[c["math"]]
            if cost <= 2e12:
                return c
    while True:
        c = dict(kind="conv", B=_log_int(rng, 1, 256), H=rng.randint(4, 32),
                 c_in=rng.choice([1, 3, 6, 64, 64, 64, 128, 128, 192, 256, 512]),
                 c_out=rng.choice([64, 64, 64, 128, 128, 128, 256, 256, 512, 48]),
                 k=rng.choice([1, 3, 3, 3, 3, 5]), stride=rng.choice([1, 1, 1, 2]), M=rng.choice([16, 20, 32, 32, 48, 64]),
                 math=rng.choice(["bf16", "bf16", "bf16", "bf16", "bf16", "x3"]), tau=tau, bwd=bwd)
        if c["math"] == "x3" or c["c_out"] == 48:      # forms that gather the operand per tap: smaller batches
            if _conv_cost(c) > 4e10:
                continue
        if _conv_cost(c) <= 6e11:
            return c


# -- what a user has in hand ------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _layer(c):
    """Layer constants: dense and multi-spike layers on [0, 1] or [0, 1.2], conv layers the window and
    synfire penalties of layer 2 of a network."""
    tm, ts = (float(x) for x in c["tau"].split(","))
    if c["kind"] == "conv":
        w = configs.synfire_layer(2)
    else:
        w = dict(t_first=0.0, t_end=1.2 if c["kind"] == "ms" else 1.0)
    dt = (w["t_end"] - w["t_first"]) / c["M"]
    return dict(tau_v=tm, tau_I=ts, v_th=1.0, M=c["M"], t_offset=0.21 * dt, **w)


def _hw_out(c):
    return (c["H"] + 2 * (c["k"] // 2) - c["k"]) // c["stride"] + 1


def _arrays(c, seed):
    """Input spike times, weights and upstream gradient of a single layer."""
    g = _gen(seed)
    if c["kind"] == "conv":
        shape, Ho = (c["B"], c["H"], c["H"], c["c_in"]), _hw_out(c)
        t = (0.7 + 0.2 * torch.randn(shape, device="cuda", generator=g)).clamp_(0.1, 1.2)
        t.masked_fill_(torch.rand(shape, device="cuda", generator=g) < 0.25, INF)
        fan, w_shape = c["c_in"] * c["k"] ** 2, (c["c_out"], c["k"], c["k"], c["c_in"])
        out, mean = (c["B"], Ho, Ho, c["c_out"]), CONV_MEAN[c["tau"]]
    else:
        shape = (c["B"], c["n_in"]) + ((c["spikes"],) if c["kind"] == "ms" else ())
        t = torch.rand(shape, device="cuda", generator=g)
        t.masked_fill_(torch.rand(shape, device="cuda", generator=g) < (0.25 if c["kind"] == "ms" else 0.1), INF)
        if c["kind"] == "ms":
            t = t.sort(-1).values
        fan, w_shape = c["n_in"], (c["n_out"], c["n_in"])
        out = (c["B"], c["n_out"]) + ((c["spikes"],) if c["kind"] == "ms" else ())
        mean = DENSE_MEAN[c["tau"]] if c["kind"] == "dense" else 6.0 * 4.0 / c["spikes"]
    W = mean / fan + torch.randn(w_shape, device="cuda", generator=g) / math.sqrt(fan)
    up = GRAD_SCALE * torch.randn(out, device="cuda", generator=g) if c["bwd"] else None
    return t, W, up


def _norm(c):
    return 1.0 / (c["B"] * (_hw_out(c) ** 2 if c["kind"] == "conv" else 1))


def _net_cfg(c):
    return configs.config2(batch=c["B"], M=c["M"]) if c["kind"] == "mlp" else configs.syn_snn20(batch=c["B"], M=c["M"])


def prepare(c, seed):
    if c["kind"] in ("mlp", "syn20"):
        cfg = _net_cfg(c)
        n = net.DenseNet(cfg, "x3") if c["kind"] == "mlp" else net.ConvNet(cfg, with_adamw=False)
        n.set_inputs(cfg["inputs"](seed), cfg["labels"](seed + 1))
        return dict(case=c, net=n)
    t, W, up = _arrays(c, seed)
    L = _layer(c)
    p = dstd.params(L, _norm(c))
    st = dict(case=c, t=t, W=W, up=up, p=p)
    u8 = dict(dtype=torch.uint8, device="cuda")
    if c["kind"] == "conv":
        B, H, C = c["B"], c["H"], c["c_in"]
        ws = dstd.conv_workspace_bytes(B, H, H, C, c["c_out"], c["k"], c["stride"], c["k"] // 2, p, c["math"])
        Ho = _hw_out(c)
        saved, out = dstd.dense_saved_bytes(B * Ho * Ho, c["c_out"]), (B, Ho, Ho, c["c_out"])
    elif c["kind"] == "ms":
        ws = dstd.ms_workspace_bytes(c["B"], c["n_in"], c["n_out"], c["spikes"], c["spikes"], p, c["math"])
        saved, out = dstd.ms_saved_bytes(c["B"], c["n_out"], c["spikes"]), (c["B"], c["n_out"], c["spikes"])
    else:
        ws = dstd.dense_workspace_bytes(c["B"], c["n_in"], c["n_out"], p, c["math"])
        saved, out = dstd.dense_saved_bytes(c["B"], c["n_out"]), (c["B"], c["n_out"])
    if ws == 0:
        raise ValueError("the library does not take this layer")
    st.update(ws=torch.empty(ws, **u8), saved=torch.empty(saved, **u8), t_out=torch.empty(out, device="cuda"),
              pen=torch.zeros(4, device="cuda"))
    if c["bwd"]:
        st.update(g_in=torch.empty_like(t), g_W=torch.empty_like(W))
    return st


def run(s):
    c = s["case"]
    if c["kind"] in ("mlp", "syn20"):
        n = s["net"]
        if not c["bwd"]:
            n.forward()
            return dict(t_out=n.t[-1], penalty=n.penalty)
        n.forward_loss()
        n.backward()
        return dict(t_out=n.t[-1], penalty=n.penalty, loss=n.loss, g_W=n.gW)
    if c["kind"] == "conv":
        a = (c["stride"], c["k"] // 2, s["p"], c["math"])
        dstd.conv_fwd(s["t"], s["W"], *a, s["t_out"], s["saved"], s["pen"], s["ws"])
        if c["bwd"]:
            dstd.conv_bwd(s["t"], s["W"], s["t_out"], s["saved"], s["up"], *a, s["g_in"], s["g_W"], s["ws"])
    elif c["kind"] == "ms":
        dstd.dense_fwd_ms(s["t"], s["W"], s["p"], c["math"], s["t_out"], s["saved"], s["ws"])
        if c["bwd"]:
            dstd.dense_bwd_ms(s["t"], s["W"], s["t_out"], s["saved"], s["up"], s["p"], c["math"], s["g_in"], s["g_W"],
                              s["ws"])
    else:
        dstd.dense_fwd(s["t"], s["W"], s["p"], c["math"], s["t_out"], s["saved"], s["pen"], s["ws"])
        if c["bwd"]:
            dstd.dense_bwd(s["t"], s["W"], s["t_out"], s["saved"], s["up"], s["p"], c["math"], s["g_in"], s["g_W"],
                           s["ws"])
    out = dict(t_out=s["t_out"])
    if c["kind"] != "ms":
        out["penalty"] = s["pen"]
    if c["bwd"]:
        out.update(g_in=s["g_in"], g_W=s["g_W"])
    return out


# -- what a pass cannot do without ------------------------------------------------------------------

def _layer_work(positions_in, n_out_total, weights, contributions, bwd, fin=1, fout=1):
    """Bytes: spike times and weights in, spike times out (backward: upstream gradient in, both gradients
    out); flops: two grid weights per input spike and connection, per contraction."""
    b = 4 * (positions_in * fin + weights + n_out_total * fout)
    f = 4 * contributions * fin
    if bwd:
        b += 4 * (n_out_total * fout + positions_in * fin + weights)
        f *= 3
    return b, f


def work(c):
    if c["kind"] in ("mlp", "syn20"):
        B = c["B"]
        if c["kind"] == "mlp":
            sizes = [784, 800, 800, 10]
            b = 4 * B * (784 + 10)
            f = 0
            for l in range(3):
                n = sizes[l] * sizes[l + 1]
                b += 4 * n * (2 if c["bwd"] else 1)
                f += 4 * B * n * ((3 if l else 2) if c["bwd"] else 1)
            return {"bytes": b, "flops": f}
        b, f = 4 * B * (28 * 28 + 10), 0
        spec = [(1, 64, 28, 28)]
        for n, H, kinds in ((64, 28, ("SD2", "SD1")), (128, 14, ("SD2", "SD1")), (256, 7, ("SD2", "SD1"))):
            for kind in kinds:
                out = (2 * n, -(-H // 2)) if kind == "SD1" else (n, H)
                spec += [(n, n, H, H), (n, n, H, H), (2 * n, out[0], H, out[1])]
        for ci, co, _, ho in spec:
            b += 4 * 9 * ci * co
            f += 4 * B * ho * ho * 9 * ci * co
        return {"bytes": b + 4 * 8192 * 10, "flops": f + 4 * B * 8192 * 10}
    if c["kind"] == "conv":
        P, Q = c["B"] * c["H"] ** 2, c["B"] * _hw_out(c) ** 2
        n = c["k"] ** 2 * c["c_in"] * c["c_out"]
        b, f = _layer_work(P * c["c_in"], Q * c["c_out"], n, Q * n, c["bwd"])
    else:
        s = c.get("spikes", 1)
        n = c["n_in"] * c["n_out"]
        b, f = _layer_work(c["B"] * c["n_in"], c["B"] * c["n_out"], n, c["B"] * n, c["bwd"], s, s)
    return {"bytes": b, "flops": f}


# -- the same in 64 bits ----------------------------------------------------------------------------

class _Layer64:
    """One layer's arithmetic in float64 (grid, kernels, binning, solve and gradient of the spike times)."""

    def __init__(self, L, norm):
        f32 = lambda x: float(np.float32(x))
        self.M = L["M"]
        self.av, self.ai = (0.0 if math.isinf(L[k]) else 1.0 / f32(L[k]) for k in ("tau_v", "tau_I"))
        self.t0, self.t1, off = f32(L["t_first"]), f32(L["t_end"]), f32(L["t_offset"])
        self.dt = (self.t1 - self.t0) / self.M
        self.t0 -= off
        self.th = f32(L["v_th"])
        self.norm = f32(norm)
        self.head, self.tail = f32(L.get("t_head_l", 0.0)), f32(L.get("t_tail_l", 0.0))
        self.gh, self.gt, self.gq = (f32(L.get(k, 0.0)) for k in ("gamma_head", "gamma_tail", "gamma_q"))
        self.energy = self.doubt = 0.0

    def tangential(self):
        """Whether neurons that only just reach the threshold rule the gradients taken so far. A spike's factor
        1 / v' is uncertain by about v'' dv / v'^2 of itself when the potential is, as in 32 bits, off by dv:
        such gradients have no value in 64 bits that an implementation in 32 can be held to."""
        return bool(self.doubt > 1e-6 * self.energy)

    def K(self, x):
        """Potential at x >= 0 after a unit input at 0."""
        if self.av == self.ai:
            return x * torch.exp(-self.av * x)
        return (torch.exp(-self.av * x) - torch.exp(-self.ai * x)) / (self.ai - self.av)

    def dK(self, x):
        return torch.exp(-self.ai * x) - self.av * self.K(x)

    def weights(self, t):
        """Grid index k of each spike, its weights at T_k and T_{k+1}, and their derivatives."""
        u = (t.double() - self.t0) / self.dt
        k = torch.floor(u)
        live = torch.isfinite(t) & (k >= -1) & (k < self.M)
        x = torch.where(live, (1.0 - (u - k)) * self.dt, torch.zeros_like(u))       # to T_{k+1}
        dt = torch.tensor(self.dt, dtype=torch.float64, device=t.device)
        a, da = self.K(x) / self.K(dt), -self.dK(x) / self.K(dt)
        e = torch.exp(-self.ai * dt)
        b, db = torch.exp(-self.ai * x) - a * e, self.ai * torch.exp(-self.ai * x) - da * e
        return torch.where(live, k, torch.full_like(k, -3)).long(), [v * live for v in (a, b, da, db)]

    def binned(self, t, which=(0, 1), round_to=None):
        """[..., N] -> [..., M, N]; which = (2, 3) for the derivatives."""
        k, w = self.weights(t)
        s = torch.zeros(t.shape[:-1] + (self.M + 2, t.shape[-1]), dtype=torch.float64, device=t.device)
        for d, j in enumerate(which):
            v = w[j] if round_to is None else w[j].to(round_to).double()
            at = k + d
            ok = (at >= 0) & (at < self.M)
            s.scatter_add_(-2, torch.where(ok, at, torch.full_like(at, self.M)).unsqueeze(-2), (v * ok).unsqueeze(-2))
        return s[..., :self.M, :]

    def _first(self, v, i, s0, s1):
        """First s in [s0, s1) at which the free potential from (v, i) at s0 reaches the threshold, else inf."""
        f = lambda s: v * torch.exp(-self.av * (s - s0)) + i * self.K(s - s0)
        df = lambda s: -self.av * v * torch.exp(-self.av * (s - s0)) + i * self.dK(s - s0)
        lo, hi = s0, torch.full_like(s0, s1)
        peak = (df(lo) > 0) & (df(hi) < 0)
        a, b = lo, hi
        for _ in range(40):
            m = 0.5 * (a + b)
            up = df(m) > 0
            a, b = torch.where(up, m, a), torch.where(up, b, m)
        top = torch.where(peak, a, hi)
        hit = f(top) >= self.th
        a, b = lo, top
        for _ in range(40):
            m = 0.5 * (a + b)
            up = f(m) >= self.th
            a, b = torch.where(up, a, m), torch.where(up, m, b)
        return torch.where(hit, 0.5 * (a + b), torch.full_like(lo, INF))

    def spikes(self, what, most=1):
        """what [P, M] -> spike times [P, most], ascending, inf after the last."""
        P = what.shape[0]
        t = torch.full((P, most), INF, dtype=torch.float64, device=what.device)
        v, i = (torch.zeros(P, dtype=torch.float64, device=what.device) for _ in range(2))
        n = torch.zeros(P, dtype=torch.long, device=what.device)
        bound = torch.tensor(self.dt, dtype=torch.float64, device=what.device)
        kmax = max(float(self.K(bound * x / 16)) for x in range(1, 17)) * 1.01
        for q in range(self.M):
            i = i + what[:, q]
            s = torch.zeros_like(v)
            at = torch.nonzero((n < most) & (v.clamp(min=0) + i.clamp(min=0) * kmax >= self.th)).squeeze(1)
            while at.numel():
                r = self._first(v[at], i[at], s[at], self.dt)
                f = torch.isfinite(r)
                at, r = at[f], r[f]
                t[at, n[at]] = self.t0 + q * self.dt + r
                i[at] = i[at] * torch.exp(-self.ai * (r - s[at]))
                v[at], s[at] = 0.0, r
                n[at] += 1
                at = at[n[at] < most]
            d = self.dt - s
            v, i = v * torch.exp(-self.av * d) + i * self.K(d), i * torch.exp(-self.ai * d)
        return t

    def g_what(self, what, t, g):
        """Gradient of sum(g t) by the implicit function theorem: one differentiable Newton step at the spikes."""
        T = self.t0 + self.dt * torch.arange(self.M, dtype=torch.float64, device=what.device)
        w = what.detach().requires_grad_(True)
        total, prev = 0.0, None
        for k in range(t.shape[1]):
            fired = torch.isfinite(t[:, k])
            tk = torch.where(fired, t[:, k], torch.zeros_like(t[:, k])).detach()
            x = tk[:, None] - T
            on = (x >= 0) & fired[:, None]
            since = torch.zeros_like(x, dtype=torch.bool)
            if prev is not None:
                y = prev[:, None] - T
                since = (y >= 0) & on
            new = on & ~since
            x0 = torch.where(new, x, torch.zeros_like(x))
            f = (torch.where(new, self.K(x0), torch.zeros_like(x)) * w).sum(1)
            df = (torch.where(new, self.dK(x0), torch.zeros_like(x)) * w.detach()).sum(1)
            if prev is not None:
                i = (torch.where(since, torch.exp(-self.ai * y.clamp(min=0)), torch.zeros_like(x)) * w).sum(1)
                d = (tk - prev).clamp(min=0)
                f, df = f + i * self.K(d), df + i.detach() * self.dK(d.detach())
            df = df.clamp(min=1e-6 * self.th / self.dt)
            c2 = torch.where(fired, g[:, k] / df, torch.zeros_like(f)).detach() ** 2
            self.energy += c2.sum()
            self.doubt += (c2 * (1e-5 / df.detach() ** 2) ** 2).sum()
            tk = torch.where(fired, tk - (f - self.th) / df, tk)
            total = total + (torch.where(fired, g[:, k], torch.zeros_like(f)) * tk).sum()
            prev = torch.where(fired, tk, torch.full_like(tk, -1e3))
        return torch.autograd.grad(total, w)[0]

    def penalty_grad(self, t):
        fired = torch.isfinite(t)
        x = torch.where(fired, t, torch.zeros_like(t))
        return self.norm * 2 * (self.gh * (x - self.head) * (fired & (x < self.head)) +
                                self.gt * (x - self.tail) * (fired & (x > self.tail)))

    def penalty(self, t, rowsum):
        """t [..., N]: (norm T, gamma_Q norm Q, silent, firing)."""
        fired = torch.isfinite(t)
        x = torch.where(fired, t, torch.zeros_like(t))
        T = self.gh * ((x - self.head) ** 2)[fired & (x < self.head)].sum() + \
            self.gt * ((x - self.tail) ** 2)[fired & (x > self.tail)].sum()
        silent = (~fired).reshape(-1, t.shape[-1]).double().sum(0)
        return torch.stack([self.norm * T, -self.gq * self.norm * (silent * rowsum).sum(), silent.sum(),
                            fired.double().sum()])


def _dense64(z, t_in, W, rnd, most, up):
    """A dense layer: spikes [B, N_out, most], and a function of the upstream gradient giving (g_in, g_W)."""
    Wd = W.to(rnd).double() if rnd else W.double()
    single = t_in.dim() == 2
    tt = t_in.unsqueeze(-1) if single else t_in
    B, M, n_out = t_in.shape[0], z.M, W.shape[0]
    s = sum(z.binned(tt[..., f], round_to=rnd) for f in range(tt.shape[-1]))           # [B, M, N_in]
    what = torch.matmul(s, Wd.t()).transpose(1, 2).reshape(B * n_out, M)
    t = z.spikes(what, most).reshape(B, n_out, most)

    def back(g):
        g = g.double().reshape(B * n_out, most)
        if single:
            g = g + z.penalty_grad(t).reshape(B * n_out, most)
        gw = z.g_what(what, t.reshape(B * n_out, most), g).reshape(B, n_out, M)
        g_W = torch.einsum("bom,bmi->oi", gw, s)
        if single:
            g_W = g_W - z.gq * z.norm * (~torch.isfinite(t[..., 0])).double().sum(0)[:, None]
        gS = torch.einsum("bom,oi->bmi", gw, Wd)
        g_in = torch.stack([(gS * z.binned(tt[..., f], (2, 3))).sum(1) for f in range(tt.shape[-1])], -1)
        return (g_in[..., 0] if single else g_in), g_W
    return t, back


def _conv64(c, t_in, W, rnd, z, up):
    """A conv layer, some images at a time."""
    k, st, pad = c["k"], c["stride"], c["k"] // 2
    B, H, _, C = t_in.shape
    O, Ho, M = c["c_out"], _hw_out(c), z.M
    W4 = (W.to(rnd).double() if rnd else W.double()).permute(0, 3, 1, 2).reshape(O, -1)
    step = max(1, int(1e9 // (M * Ho * Ho * max(O, C * k * k))))
    ts, gi, gW = [], [], torch.zeros_like(W4)
    for b in range(0, B, step):
        t = t_in[b:b + step]
        n = t.shape[0]
        img = lambda v: v.transpose(1, 2).reshape(n * M, C, H, H)                       # [n, M, HWC] -> planes
        flat = t.permute(0, 3, 1, 2).reshape(n, -1)
        s = z.binned(flat, round_to=rnd).reshape(n * M, C, H, H)
        cols = F.unfold(s, k, padding=pad, stride=st)                                   # [nM, Ckk, L]
        what = torch.matmul(W4, cols).reshape(n, M, O, Ho * Ho).permute(0, 3, 2, 1).reshape(-1, M)
        to = z.spikes(what)
        ts.append(to.reshape(n, Ho, Ho, O))
        if up is None:
            continue
        g = up[b:b + step].double().reshape(-1, 1) + z.penalty_grad(to)
        gw = z.g_what(what, to, g).reshape(n, Ho * Ho, O, M).permute(0, 3, 2, 1).reshape(n * M, O, Ho * Ho)
        gW += torch.matmul(gw.transpose(0, 1).reshape(O, -1), cols.transpose(1, 2).reshape(-1, cols.shape[1]))
        gs = F.fold(torch.matmul(W4.t(), gw), (H, H), k, padding=pad, stride=st).reshape(n, M, -1)
        gi.append((gs * z.binned(flat, (2, 3))).sum(1).reshape(n, C, H, H).permute(0, 2, 3, 1))
    t = torch.cat(ts)
    out = dict(t_out=t, penalty=z.penalty(t, W.double().reshape(O, -1).sum(1)))
    if up is not None:
        gW = gW.reshape(O, C, k, k).permute(0, 2, 3, 1)
        silent = (~torch.isfinite(t)).reshape(-1, O).double().sum(0)
        if z.tangential():
            return dict(out, g_in=None, g_W=None)
        out.update(g_in=torch.cat(gi), g_W=gW - z.gq * z.norm * silent[:, None, None, None])
    return out


def _mlp64(c, seed):
    cfg = _net_cfg(c)
    t = torch.as_tensor(cfg["inputs"](seed), dtype=torch.float32, device="cuda")
    labels = torch.as_tensor(cfg["labels"](seed + 1), device="cuda")
    B, backs, pens = c["B"], [], []
    for L in cfg["layers"]:
        W = torch.tensor(L["W"], dtype=torch.float32, device="cuda")
        z = _Layer64(L, 1.0 / B)
        to, back = _dense64(z, t, W, None, 1, None)
        t = to[..., 0]
        backs.append((back, z))
        pens.append(z.penalty(t, W.double().sum(1)))
    out = dict(t_out=t, penalty=torch.stack(pens))
    if c["bwd"]:
        fired = torch.isfinite(t)
        soft = float(np.float32(cfg["tau_soft"]))
        x = -torch.where(fired, t, torch.full_like(t, float(np.float32(cfg["layers"][-1]["t_end"])))) / soft
        kap = F.one_hot(labels.long(), t.shape[1]).double()
        loss = -(torch.log_softmax(x, 1) * kap).sum() / B
        g = torch.where(fired, -(torch.softmax(x, 1) - kap) / soft / B, torch.zeros_like(x))
        gW, lost = [], False
        for back, z in reversed(backs):
            g, gw = back(g)
            lost = lost or z.tangential()
            gW.insert(0, None if lost else gw)
        out.update(loss=torch.stack([loss, torch.zeros_like(loss)]), g_W=gW)
    return out


def exact(c, seed):
    if c["kind"] == "syn20":
        return None                # 20 bf16 layers deep: no value in 64 bits to hold them to
    if 2.0 * (3 if c["bwd"] else 1) * work(c)["flops"] / (6 if c["bwd"] else 2) * c["M"] > 1e13:
        return None                # over 20 seconds of 64-bit arithmetic
    if c["kind"] == "mlp":
        return _mlp64(c, seed)
    t, W, up = _arrays(c, seed)
    z = _Layer64(_layer(c), _norm(c))
    rnd = torch.bfloat16 if c["math"] == "bf16" else None
    if c["kind"] == "conv":
        return _conv64(c, t, W, rnd, z, up)
    to, back = _dense64(z, t, W, rnd, c.get("spikes", 1), up)
    out = dict(t_out=to if c["kind"] == "ms" else to[..., 0])
    if c["kind"] != "ms":
        out["penalty"] = z.penalty(out["t_out"], W.double().sum(1))
    if c["bwd"]:
        g_in, g_W = back(up)
        out.update(g_in=None, g_W=None) if z.tangential() else out.update(g_in=g_in, g_W=g_W)
    return out
