"""What the speed of this library is measured on: optimizer steps, layer statistics and
gradient-scale updates over the parameter sets of this repository, through the calls a training
program makes.

A case is a dict of plain values:

  call      "step" (one optimizer step), "stats" (tula_layer_stats) or "scale"
            (tula_ags_update_scale)
  set       a parameter set of ``workloads`` ("resnet20" ... "vgg16"), or "log": `tensors` 1-D
            tensors with sizes log-uniform in [64, hi], odd ones among them (the recipe of the
            stress set)
  K         replica gradients
  layout    "padded": every tensor at a 256-byte boundary, as separate allocations lie;
            "buckets": the gradients lie back to back in one flat buffer per replica (the
            buckets of a data-parallel trainer), weights and momentum are padded;
            "packed": every role lies back to back in one flat buffer
  rule      step: "ags", "none", "static" or "lars"
  refresh   step: UpdateGradScale after the update
  element   step, scale: one gradscale per element
  momentum  step: with momentum buffers
  stats     step: with the per-layer statistics
  plan      step: through a plan, or through tula_ags_step
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_18112_gb300 import tula_ags as T
from paper_2603_18112_gb300 import workloads as W

LR, MU, WD = 0.1, 0.9, 5e-4
DELTA, EPS, STATIC_S, LARS_TRUST = 0.5, 1e-8, 1.5, 1e-3
RULES = {"ags": T.TULA_RULE_AGS, "none": T.TULA_RULE_NONE, "static": T.TULA_RULE_STATIC,
         "lars": T.TULA_RULE_LARS}


def _step(**kw):
    case = {"call": "step", "layout": "padded", "rule": "ags", "refresh": False, "element": False,
            "momentum": True, "stats": True, "plan": True}
    case.update(kw)
    return case


def listed():
    return [
        # The smallest model: one worker's own gradient, a few microseconds of work, so that
        # launches and latency are what a training loop sees.
        _step(name="resnet20_k1", set="resnet20", K=1),
        # A model of many small layers (norms, biases, thin convolutions): little data, many
        # tensors.
        _step(name="small_layers_k4", set="log", tensors=1024, hi=4096, K=4),
        # An ordinary mid-size model, tens of microseconds.
        _step(name="resnet18_k4", set="resnet18", K=4),
        # The benchmark's own set: Algorithm 1 every iteration.
        _step(name="resnet50_k8", set="resnet50", K=8),
        # The prior-art rule, whose norms feed the step.
        _step(name="resnet50_k8_lars", set="resnet50", K=8, rule="lars"),
        # Algorithm 1 as it is written, one gradscale per element, without momentum or records.
        _step(name="resnet50_k8_element", set="resnet50", K=8, element=True, momentum=False,
              stats=False),
        # A worker count that is no power of two.
        _step(name="resnet50_k6", set="resnet50", K=6),
        # Gradients as views into flat buckets, with tensor sizes that are not multiples of four:
        # most views start off a 16-byte boundary.
        _step(name="odd_sizes_k4_buckets", set="log", tensors=128, hi=1 << 20, K=4,
              layout="buckets"),
        # One large fully connected layer beside small ones; the step after which UpdateGradScale
        # runs.
        _step(name="vgg16_k8_refresh", set="vgg16", K=8, refresh=True),
        # The largest: thousands of tensors of very unequal sizes, sixteen workers.
        _step(name="stress_k16", set="log", tensors=4096, hi=1 << 18, K=16),
        # Monitoring without a step: the norms of every layer.
        {"name": "vgg16_k4_stats", "call": "stats", "set": "vgg16", "K": 4, "layout": "padded"},
        # UpdateGradScale from a separate small-batch gradient, element by element.
        {"name": "resnet50_scale_element", "call": "scale", "set": "resnet50", "K": 1,
         "layout": "padded", "element": True},
    ]


MOST_BYTES = 4e9      # of a drawn case; the largest listed one moves about 11 GB
MOST_ODD_BYTES = 1e9  # and of one whose tensors lie back to back


def draw(rng):
    call = rng.choices(("step", "stats", "scale"), (8, 1, 1))[0]
    layout = rng.choices(("padded", "buckets", "packed"), (3, 1, 1))[0]
    K = 1 if call == "scale" else rng.choice((1, 2, 3, 4, 5, 6, 7, 8, 8, 10, 12, 16))
    case = {"call": call, "layout": layout, "K": K}
    if call == "step":
        case = _step(**case)
        case["rule"] = rng.choices(("ags", "none", "static", "lars"), (6, 1, 1, 2))[0]
        case["momentum"] = rng.random() < 0.8
        case["stats"] = rng.random() < 0.8
        case["plan"] = rng.random() < 0.8
        if case["rule"] == "ags":
            case["element"] = rng.random() < 0.15
            case["refresh"] = K > 1 and not case["element"] and rng.random() < 0.3
    elif call == "scale":
        case["element"] = rng.random() < 0.5
    if rng.random() < 0.25:
        case["set"] = rng.choice(("resnet20", "resnet18", "resnet50", "vgg16"))
        if work(case)["bytes"] <= MOST_BYTES:
            return case
    case["set"] = "log"
    most = MOST_BYTES if layout == "padded" else MOST_ODD_BYTES
    while True:
        case["tensors"] = int(round(math.exp(rng.uniform(0.0, math.log(4096)))))
        case["hi"] = int(round(math.exp(rng.uniform(math.log(256), math.log(1 << 24)))))
        if work(case)["bytes"] <= most:
            return case


# --------------------------------------------------------------------------------------------
# Shapes and inputs
# --------------------------------------------------------------------------------------------

def _params(case):
    if case["set"] != "log":
        return W.param_set(case["set"])
    n, hi = case["tensors"], case["hi"]
    rng = np.random.default_rng([n, hi])
    sizes = np.rint(np.exp(rng.uniform(math.log(64), math.log(hi), size=n))).astype(np.int64)
    ps = W.ParamSet("log")
    for s in sizes:
        ps.add((int(s),), W.KIND_NORMAL)
    return ps


def _layout(numels, padded):
    """First element of each tensor in its role's flat buffer, and the buffer's length."""
    room = [(n + 63) // 64 * 64 if padded else n for n in numels]
    ends = np.cumsum(room)
    return [int(e) - r for e, r in zip(ends, room)], int(ends[-1])


class _Inputs:
    """One role per flat buffer: w, m, g[k] (step, stats), or small and large gradients (scale).

    Weights are Kaiming-normal (norm gains 1, biases 0; N(0, 0.02) in the "log" sets), gradients
    N(0, 1e-3) times a factor per tensor, log-uniform in [0.1, 10] and shared by the replicas,
    momentum N(0, 1e-3)."""

    def __init__(self, case, seed):
        ps = _params(case)
        self.shapes, self.numels, self.n = ps.shapes, ps.numels, ps.n_tensors
        self.w_off, w_len = _layout(self.numels, case["layout"] != "packed")
        self.g_off, g_len = _layout(self.numels, case["layout"] == "padded")
        gen = torch.Generator(device="cuda").manual_seed(1 + int(seed))
        host = np.random.default_rng([int(seed), 7])

        def normal(length):
            return torch.randn(length, generator=gen, device="cuda")

        std, mean = np.zeros(self.n), np.zeros(self.n)
        for p, (shape, kind) in enumerate(zip(ps.shapes, ps.kinds)):
            if kind == W.KIND_WEIGHT:
                std[p] = math.sqrt(2.0 / float(np.prod(shape[1:])))
            elif kind == W.KIND_BN_GAMMA:
                mean[p] = 1.0
            elif kind == W.KIND_NORMAL:
                std[p] = 0.02
        factors = 1e-3 * np.exp(host.uniform(math.log(0.1), math.log(10.0), self.n))
        g_fac = self._spread(factors, self.g_off, g_len)
        K = case["K"]
        self.g = [normal(g_len).mul_(g_fac) for _ in range(K)]
        if case["call"] == "scale":
            # a sub-batch's gradient: the large batch's with more noise
            self.small = normal(g_len).mul_(g_fac).add_(self.g[0])
            return
        self.w = normal(w_len).mul_(self._spread(std, self.w_off, w_len))
        self.w.add_(self._spread(mean, self.w_off, w_len))
        if case["call"] == "step":
            self.m = normal(w_len).mul_(1e-3) if case["momentum"] else None
            # a gradscale per tensor, or per element, as a run some epochs old holds it
            self.scale = torch.rand(self.n, generator=gen, device="cuda").mul_(math.sqrt(K)).add_(0.5)
            self.scale_elem = (torch.rand(w_len, generator=gen, device="cuda").mul_(math.sqrt(K))
                               if case["element"] else None)
            # the last iteration's |G|^2, about as large as this one's: Delta is about 0.2
            total = 0.0
            for o in range(0, g_len, 1 << 25):
                mean = sum(g[o:o + (1 << 25)] for g in self.g) / K
                total += float(mean.double().square_().sum())
            self.g2_prev = 1.25 * total

    def _spread(self, values, off, length):
        """One value per tensor, repeated over the tensor's elements; 0 in the padding after it."""
        both, counts = np.zeros((self.n, 2), np.float32), np.zeros((self.n, 2), np.int64)
        both[:, 0], counts[:, 0] = values, self.numels
        counts[:, 1] = np.append(off[1:], length) - np.array(off) - counts[:, 0]
        return torch.repeat_interleave(torch.from_numpy(both.ravel()).cuda(),
                                       torch.from_numpy(counts.ravel()).cuda(), output_size=length)

    def views(self, flat, off):
        return [flat[o:o + n].view(s) for o, n, s in zip(off, self.numels, self.shapes)]


# --------------------------------------------------------------------------------------------
# The calls
# --------------------------------------------------------------------------------------------

def prepare(case, seed):
    x = _Inputs(case, seed)
    st = {"case": case, "x": x}
    if case["call"] == "step":
        step = T.AGSOptimizerStep(
            x.views(x.w, x.w_off), [x.views(g, x.g_off) for g in x.g],
            x.views(x.m, x.w_off) if x.m is not None else None, rule=RULES[case["rule"]],
            granularity=T.TULA_SCALE_PER_ELEMENT if case["element"] else T.TULA_SCALE_PER_TENSOR,
            delta=DELTA, eps=EPS, static_s=STATIC_S, lars_trust=LARS_TRUST, scale=x.scale,
            scale_elem=x.views(x.scale_elem, x.w_off) if case["element"] else None,
            stats=case["stats"], plan=case["plan"])
        # a run in its fifth iteration
        step.state.copy_(torch.tensor([x.g2_prev, 4.0, 0.2, 1.0], dtype=torch.float64))
        st["step"] = step
        st["mu"] = MU if case["momentum"] else 0.0
        out = {"w": x.w, "state": step.state, "g": x.g[0]}
        if x.m is not None:
            out["m"] = x.m
        if case["stats"]:
            out["stats"] = step.stats
        if case["refresh"]:
            out["scale"] = step.scale
        st["out"] = out
    elif case["call"] == "stats":
        st["w"] = x.views(x.w, x.w_off)
        st["g"] = [x.views(g, x.g_off) for g in x.g]
        st["workspace"] = T.new_workspace(x.numels, case["K"])
        st["out"] = torch.zeros(x.n, T.TULA_STATS_LEN, dtype=torch.float64, device="cuda")
    else:
        st["small"] = x.views(x.small, x.g_off)
        st["large"] = x.views(x.g[0], x.g_off)
        hp = T.tula_ags_default_hparams(8)
        if case["element"]:
            st["out"] = torch.zeros_like(x.small)
            st["ptrs"] = T._tensor_ptrs(x.views(st["out"], x.g_off))
            hp.granularity = T.TULA_SCALE_PER_ELEMENT
            hp.scale_elem = T.ctypes.cast(st["ptrs"], T.c_void_p).value
        else:
            st["out"] = torch.zeros(x.n, dtype=torch.float32, device="cuda")
            st["workspace"] = T.new_workspace(x.numels, 1)
            hp.scale = st["out"].data_ptr()
            hp.workspace = st["workspace"].data_ptr()
            hp.workspace_bytes = st["workspace"].numel()
        st["hp"] = hp
    torch.cuda.synchronize()
    return st


def run(state):
    case = state["case"]
    if case["call"] == "step":
        state["step"].step(LR, state["mu"], WD, refresh_scale=case["refresh"])
    elif case["call"] == "stats":
        T.tula_layer_stats(state["w"], state["g"], state["out"], state["workspace"])
    else:
        T.tula_ags_update_scale(state["small"], state["large"], state["hp"])
    return state["out"]


def work(case):
    """Every gradient, weight and momentum element read once; weights, momentum, the mean (K > 1,
    over replica 0) and element-wise gradscales written once."""
    N, K = sum(_params(case).numels), case["K"]
    if case["call"] == "scale":
        return {"bytes": (12.0 if case["element"] else 8.0) * N, "flops": 4.0 * N}
    if case["call"] == "stats":
        return {"bytes": 4.0 * (K + 1) * N, "flops": (K + 6.0) * N}
    per = 4 * K + 8 + (4 if K > 1 else 0) + (8 if case["momentum"] else 0)
    per += 4 if case["element"] else 0
    return {"bytes": float(per) * N, "flops": (K + 14.0) * N}


def tolerance(case):
    """Element-wise results are a few fp32 operations (6e-8 each), the default norms fp32 sums
    within a tile: outputs lie up to 8.3e-8 from exact() (the largest, w, m and the mean of
    sixteen replicas), so another order of the same sums may be four times that from these."""
    return {"rel": 4e-7}


# --------------------------------------------------------------------------------------------
# The same in 64 bits
# --------------------------------------------------------------------------------------------

def _segments(flat, off, numels):
    """Squared norms of the tensors of a flat fp64 buffer."""
    return torch.stack([flat[o:o + n].square().sum() for o, n in zip(off, numels)])


def exact(case, seed):
    x = _Inputs(case, seed)
    K = case["K"]
    if case["call"] == "scale":
        small, large = x.small.double(), x.g[0].double()
        s_max = float(np.float32(math.sqrt(8.0)))
        eps = float(np.float32(EPS))
        if case["element"]:
            out = torch.zeros_like(small)
            q = (small / (large + eps)).abs_().clamp_(max=s_max)
            for o, n in zip(x.g_off, x.numels):
                out[o:o + n] = q[o:o + n]
            return out
        ns = _segments(small, x.g_off, x.numels).sqrt()
        nl = _segments(large, x.g_off, x.numels).sqrt()
        return (ns / (nl + eps)).clamp(max=s_max)
    mean = x.g[0].double()
    for g in x.g[1:]:
        mean += g
    mean /= K
    g_sq = _segments(mean, x.g_off, x.numels)
    g0_sq = _segments(x.g[0].double(), x.g_off, x.numels)
    w_sq = _segments(x.w.double(), x.w_off, x.numels)
    ng, nw = g_sq.sqrt(), w_sq.sqrt()
    ratio = torch.where(g_sq > 0, nw / ng, torch.zeros_like(ng))
    zero = torch.zeros_like(ng)
    if case["call"] == "stats":
        return torch.stack([w_sq, g_sq, g0_sq, nw, ng, ratio, zero, zero], 1)

    eps, s_max = float(np.float32(EPS)), float(np.float32(math.sqrt(K)))
    g2 = float(g_sq.sum())
    delta = abs((g2 - x.g2_prev) / x.g2_prev)
    scaled = delta < DELTA
    rule = case["rule"]
    if rule == "lars":
        coef = torch.where((w_sq > 0) & (g_sq > 0), float(np.float32(LARS_TRUST)) * ratio, zero + 1)
    elif rule == "static" and scaled:
        coef = zero + STATIC_S
    elif rule == "ags" and scaled and not case["element"]:
        coef = x.scale.double()
    else:
        coef = zero + 1
    lr, mu, wd = (float(np.float32(v)) for v in (LR, MU, WD))
    w, m = x.w.double(), x.m.double() if x.m is not None else None
    for p, (o, q, n) in enumerate(zip(x.w_off, x.g_off, x.numels)):
        c = x.scale_elem[o:o + n].double() if case["element"] and scaled else coef[p]
        ws = w[o:o + n]
        d = mean[q:q + n] * c + ws * wd
        if m is not None:
            m[o:o + n].mul_(mu).add_(d)
            d = m[o:o + n]
        ws -= lr * d
    state = torch.tensor([g2, 5.0, delta, float(scaled)], dtype=torch.float64)
    # the padding of replica 0 is not the library's to write
    out_g = x.g[0].double()
    for o, n in zip(x.g_off, x.numels):
        out_g[o:o + n] = mean[o:o + n]
    out = {"w": w, "state": state, "g": out_g if K > 1 else x.g[0].double()}
    if m is not None:
        out["m"] = m
    scale = x.scale.double()
    if case["refresh"]:
        scale = (g0_sq.sqrt() / (ng + eps)).clamp(max=s_max)
        out["scale"] = scale
    if case["stats"]:
        col = torch.full_like(ng, math.nan if scaled else 1.0) if case["element"] else coef
        out["stats"] = torch.stack([w_sq, g_sq, g0_sq, nw, ng, ratio, col, scale], 1)
    return out
