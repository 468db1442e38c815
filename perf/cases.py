"""The work that a training run with this library has it do, as cases that can be timed one by one.

Kinds of cases
  conv         one convolution layer outside a graph: pt_conv_fwd, pt_conv_dgrad (unless it is the first layer) and pt_conv_wgrad
  layer        one convolution with its batch norm, ReLU and residual: forward with the statistics taken by the convolution,
               then the whole backward of the layer from saved activations
  step         harness.TrainStep.step(): detection, plan, compaction gather, every layer's forward / data / weight gradient and
               the group-lasso SGD step, replayed from a CUDA graph
  lasso        the group-lasso momentum-SGD step over all layers of a pruned network, in the plain or in the carried form
  reconfigure  detection, plan and gather of a network whose groups went to zero, into the smaller one
  gate         channel gating of one node tensor: gather at a branch's entry, scatter-add with ReLU at its merge point

Inputs are drawn on the GPU from the seed: activations max(N(0,1), 0), upstream gradients N(0,1) * 2^-6, weights
N(0, sqrt(2 / fan_in)), momenta and stand-alone gradients N(0, 1e-3).
"""
import math

import numpy as np
import torch

from paper_1901_09290_b200 import binding as B
from paper_1901_09290_b200 import harness
from paper_1901_09290_b200 import workloads as W

LAM, LR, MU = 1e-4, 0.1, 0.9


# ------------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call a user makes: a CIFAR-sized layer with ragged channels, small batch; latency and launches
        dict(name="conv tiny 13-27 16x16 b8", kind="conv", N=8, H=16, C=13, K=27, R=3, stride=1, first=False),
        # the first layer of every ImageNet ResNet; it has no data gradient
        dict(name="conv stem 7x7/2 224 b64", kind="conv", N=64, H=224, C=3, K=55, R=7, stride=2, first=True),
        # the wide ragged 1x1 at the entry of a pruned ImageNet bottleneck, after the first reconfigurations
        dict(name="conv 1x1 931-213 14x14 b64", kind="conv", N=64, H=14, C=931, K=213, R=1, stride=1, first=False),
        # the downsampling 3x3 at the head of a pruned stage
        dict(name="conv 3x3/2 106-103 56x56 b64", kind="conv", N=64, H=56, C=106, K=103, R=3, stride=2, first=False),
        # the last layer of a pruned bottleneck as a chained network runs it: batch norm, residual add, ReLU, both directions
        dict(name="layer 1x1 77-371 28x28 b64", kind="layer", N=64, H=28, C=77, K=371, R=1, stride=1, residual=True),
        # a whole training step of the CIFAR ResNet-32 after pruning: many small launches
        dict(name="step resnet32 b128", kind="step", net="resnet32", N=128, draw="random", keep=0.65, keep_seed=W.BASE_SEED + 2),
        # a whole training step of the pruned ImageNet ResNet-50 (60 % of the dense FLOPs): the headline workload
        dict(name="step resnet50 0.60 b64", kind="step", net="resnet50", N=64, draw="staged", keep=0.60, keep_seed=W.BASE_SEED + 4),
        # late in training: a much smaller model, and the mini-batch grown into the memory that this freed
        dict(name="step resnet50 keep0.3 b256", kind="step", net="resnet50", N=256, draw="uniform", keep=0.3, keep_seed=0),
        # the optimiser alone, as a user's own training loop calls it after its backward pass
        dict(name="lasso resnet50 0.60", kind="lasso", net="resnet50", draw="staged", keep=0.60, keep_seed=W.BASE_SEED + 4, carried=False),
        # the same for a small network, in the form that leaves the next step's norms behind
        dict(name="lasso carried resnet32", kind="lasso", net="resnet32", draw="random", keep=0.65, keep_seed=W.BASE_SEED + 2, carried=True),
        # a reconfiguration between epochs: dense ResNet-50 with 40 % of its work gone to zero
        dict(name="reconfigure resnet50 0.60", kind="reconfigure", net="resnet50", draw="staged", keep=0.60, keep_seed=W.BASE_SEED + 4),
        # channel gating around a stage-1 branch, where the node tensor is largest
        dict(name="gate 211 of 222 56x56 b64", kind="gate", N=64, H=56, C=222, S=211),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _one(rng):
    kind = rng.choice(["conv", "conv", "conv", "layer", "layer", "step", "step", "lasso", "reconfigure", "gate"])
    if kind in ("conv", "layer"):
        N = _log(rng, 4, 256)
        if kind == "conv" and rng.random() < 0.1:
            big = rng.random() < 0.5
            return dict(kind="conv", N=N, H=224 if big else 32, C=3, K=rng.randint(8, 64), R=7 if big else 3, stride=2 if big else 1, first=True)
        R = rng.choice([1, 1, 3])
        top = 2048 if R == 1 else 512
        H = rng.choice([7, 8, 14, 16, 28, 32, 56, rng.randint(7, 56)])
        C, K = _log(rng, 8, top), _log(rng, 8, top)
        stride = rng.choice([1, 1, 1, 2])
        if kind == "conv":
            return dict(kind="conv", N=N, H=H, C=C, K=K, R=R, stride=stride, first=False)
        return dict(kind="layer", N=N, H=H, C=C, K=K, R=R, stride=stride, residual=rng.random() < 0.5)
    if kind == "gate":
        C = _log(rng, 32, 2048)
        return dict(kind="gate", N=_log(rng, 4, 256), H=rng.choice([7, 14, 28, 56, rng.randint(7, 56)]), C=C, S=max(8, int(C * rng.uniform(0.5, 1.0))))
    net = rng.choice(["resnet50", "resnet50", "resnet32", "vgg11", "vgg13"])
    c = dict(kind=kind, net=net, draw=rng.choice(["staged", "uniform", "random"]), keep=round(rng.uniform(0.3, 0.9), 3), keep_seed=rng.randint(1, 1 << 30))
    if kind == "step":
        c["N"] = 8 * _log(rng, 4, 32)
    if kind == "lasso":
        c["carried"] = rng.random() < 0.5
    return c


def draw(rng):
    """One more case of the ranges above. Channel counts, batches and image sizes are spread over what networks meet, odd ones among
    them; a case that would cost more than the largest listed one of its sort is drawn again."""
    top = [work(c) for c in listed() if c["kind"] == "step"]
    one = [work(c) for c in listed() if c["kind"] != "step"]
    while True:
        c = _one(rng)
        w, most = work(c), (top if c["kind"] == "step" else one)
        if w["bytes"] <= max(m["bytes"] for m in most) and w["flops"] <= 2e11 * (5 if c["kind"] == "step" else 1):
            return c


# ------------------------------------------------------------------------------------------------ networks
_NETS = {}


def _nets(case):
    """(dense network, kept channels per space, pruned network): shape tables, the same for every seed."""
    key = (case["net"], case["draw"], case["keep"], case["keep_seed"])
    if key not in _NETS:
        net = {"resnet50": W.resnet50, "resnet32": W.resnet32, "vgg11": lambda: W.vgg(11), "vgg13": lambda: W.vgg(13)}[case["net"]]()
        if case["draw"] == "staged":            # per-space ratios, scaled so that `keep` of the dense FLOPs are left
            counts = W.staged_keep_to_flops(net, case["keep_seed"], case["keep"])
        elif case["draw"] == "random":          # per-space ratios around `keep`
            counts = W.random_keep(net, case["keep_seed"], max(0.1, case["keep"] - 0.25), min(1.0, case["keep"] + 0.25))
        else:
            counts = W.uniform_keep(net, case["keep"])
        _NETS[key] = net, counts, W.with_sizes(net, counts)
    return _NETS[key]


def _params(net):
    return sum(l.K * l.C * l.R * l.R for l in net.layers)


class _Flat:
    """One allocation cut into views, each on a 256-byte boundary."""

    def __init__(self, shapes, dtype):
        size = torch.empty((), dtype=dtype).element_size()
        pad = 256 // size
        at, self.views = 0, []
        offs = []
        for s in shapes:
            offs.append(at)
            at += (math.prod(s) + pad - 1) // pad * pad
        self.all = torch.zeros(max(at, pad), dtype=dtype, device="cuda")
        for s, o in zip(shapes, offs):
            self.views.append(self.all[o:o + math.prod(s)].view(s))


class _Params:
    """A network's weights, momenta, gradients, shadow and masks in flat buffers, as an optimiser keeps them."""

    def __init__(self, ctx, net, gen=None, kept=None):
        L = net.layers
        full = [(l.K, l.R, l.R, l.C) for l in L]
        self.w, self.v, self.g = (_Flat(full, torch.float32) for _ in range(3))
        self.wb = _Flat([(l.K, l.R, l.R, W.pad8(l.C)) for l in L], torch.bfloat16)
        self.so, self.si = _Flat([(l.K,) for l in L], torch.float32), _Flat([(l.C,) for l in L], torch.float32)
        self.zo, self.zi = _Flat([(l.K,) for l in L], torch.uint8), _Flat([(l.C,) for l in L], torch.uint8)
        self.bn = _Flat([(4, l.K) for l in L], torch.float32)
        if gen is not None:
            for f in (self.w, self.v, self.g, self.bn):
                f.all.normal_(0.0, 1.0, generator=gen)
            self.v.all.mul_(1e-3)
            self.g.all.mul_(1e-3)
            for i, l in enumerate(L):
                self.w.views[i].mul_(math.sqrt(2.0 / (l.C * l.R * l.R)))
        if kept is not None:
            self._zero(net, kept)
        for i, l in enumerate(L):
            self.wb.views[i][..., :l.C] = self.w.views[i]
        self.layers = B.layer_array([
            B.make_layer(self.w.views[i], self.g.views[i], self.v.views[i], self.wb.views[i], l.K, l.C, l.R * l.R, W.pad8(l.C),
                         net.space_stage[l.in_space] != 0, True, self.so.views[i], self.si.views[i], self.zo.views[i], self.zi.views[i])
            for i, l in enumerate(L)])
        self.ws = torch.empty(max(256, B.pt_group_lasso_workspace_bytes(ctx, self.layers)), dtype=torch.uint8, device="cuda")
        self.reg = torch.zeros(1, dtype=torch.float64, device="cuda")
        self.graph = B.GraphHandle(net.space_sizes, net.space_fixed, list(self.layers), [(l.in_space, l.out_space) for l in L],
                                   [[b[k] for k in range(4)] for b in self.bn.views])

    def _zero(self, net, kept):
        """Every channel outside kept[space] is zero in all members of the space; two kept ones are zero in all members but the
        first (a residual node keeps such a channel for the one that still uses it)."""
        for s, size in enumerate(net.space_sizes):
            members = [(i, True) for i, l in enumerate(net.layers) if l.out_space == s] + [(i, False) for i, l in enumerate(net.layers) if l.in_space == s]
            live = torch.zeros(size, device="cuda")
            live[torch.from_numpy(kept[s]).long().cuda()] = 1.0
            rest = live.clone()
            if len(members) > 1 and len(kept[s]) > 3 and not net.space_fixed[s]:
                rest[torch.from_numpy(kept[s][:2]).long().cuda()] = 0.0
            for n, (i, out) in enumerate(members):
                m = live if n == 0 else rest
                m = m.view(-1, 1, 1, 1) if out else m
                for f in (self.w, self.v, self.g):
                    f.views[i].mul_(m)


# ------------------------------------------------------------------------------------------------ prepare
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _act(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda").clamp_(min=0).to(torch.bfloat16)


def _grad(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda").mul_(2.0 ** -6).to(torch.bfloat16)


def _conv_state(case, gen):
    N, H, C, K, R, stride = (case[k] for k in ("N", "H", "C", "K", "R", "stride"))
    P = (H + 2 * (R // 2) - R) // stride + 1
    ldx, ldy, ldw = (8 if C <= 4 else W.pad16(C)), W.pad16(K), W.pad8(C)
    s = dict(ctx=B.Context(0))
    s["d"] = B.make_conv_desc(N, H, H, C, K, R, R, stride, R // 2, ldx, ldy, ldw)
    s["x"] = torch.randn((N, H, H, ldx), generator=gen, device="cuda").to(torch.bfloat16) if case.get("first") else _act(gen, N, H, H, ldx)
    s["w"] = (torch.randn((K, R, R, ldw), generator=gen, device="cuda") * math.sqrt(2.0 / (C * R * R))).to(torch.bfloat16)
    s["dy"] = _grad(gen, N, P, P, ldy)
    s["y"], s["dx"] = torch.zeros_like(s["dy"]), torch.zeros_like(s["x"])
    s["dw"] = torch.zeros((K, R, R, C), device="cuda")
    s["ws"] = torch.empty(max(16, max(B.pt_conv_workspace_bytes(s["ctx"], s["d"], w) for w in range(3))), dtype=torch.uint8, device="cuda")
    return s


def _layer_state(case, gen):
    s = _conv_state(case, gen)
    N, K, ldy, P = case["N"], case["K"], s["d"].ldy, s["dy"].shape[1]
    s["bn"] = B.make_bn_desc(N, P, P, K, ldy)
    s["gamma"] = torch.rand(K, generator=gen, device="cuda") + 0.5
    s["beta"] = torch.rand(K, generator=gen, device="cuda") - 0.5
    s["rm"], s["rv"] = torch.zeros(K, device="cuda"), torch.ones(K, device="cuda")
    s["res"] = _act(gen, N, P, P, ldy) if case["residual"] else None
    s["mean"], s["invstd"], s["dgamma"], s["dbeta"] = (torch.zeros(K, device="cuda") for _ in range(4))
    s["a"] = torch.zeros_like(s["dy"])
    s["stats"] = torch.empty(max(4, B.pt_conv_fwd_stats_bytes(s["ctx"], s["d"]) // 4), device="cuda")
    s["bnws"] = torch.empty(max(16, B.pt_bn_workspace_bytes(s["ctx"], s["bn"])), dtype=torch.uint8, device="cuda")
    # what the forward pass of the step saved for this backward pass: convolution output, its statistics, the activation
    s["y0"] = torch.randn((N, P, P, ldy), generator=gen, device="cuda").add_(0.25).to(torch.bfloat16)
    f = s["y0"][..., :K].float()
    s["mean0"] = f.mean((0, 1, 2))
    s["invstd0"] = (f.var((0, 1, 2), unbiased=False) + 1e-5).rsqrt()
    f = f.sub_(s["mean0"]).mul_(s["invstd0"] * s["gamma"]).add_(s["beta"])
    if s["res"] is not None:
        f.add_(s["res"][..., :K])
    s["a0"] = torch.zeros_like(s["dy"])
    s["a0"][..., :K] = f.clamp_(min=0)
    s["da"] = _grad(gen, N, P, P, ldy)                    # gradient of the layer's activation
    s["dres"] = torch.zeros_like(s["dy"]) if case["residual"] else None
    s["dy"] = torch.zeros_like(s["dy"])                   # gradient of the convolution output: written by the batch norm's backward
    return s


def _step_state(case, seed):
    net, counts, pruned = _nets(case)
    ctx = B.Context(0)
    ts = harness.TrainStep(ctx, net, counts, W.choose_kept(net, counts, seed), case["N"], seed)
    # the tensors that come back, each kind in one buffer
    s = dict(ctx=ctx, ts=ts)
    s["y"] = _Flat([tuple(t.shape) for t in ts.y], torch.bfloat16)
    s["dx"] = _Flat([tuple(t.shape) for t in ts.dx[1:]], torch.bfloat16)
    ts.y, ts.dx = s["y"].views, [None] + s["dx"].views
    ts.step()
    torch.cuda.synchronize()
    ts.build_graph()
    return s


def _model_state(case, gen, seed):
    net, counts, pruned = _nets(case)
    s = dict(ctx=B.Context(0))
    if case["kind"] == "lasso":
        s["p"] = _Params(s["ctx"], pruned, gen)
        if case["carried"]:
            B.pt_group_lasso_norms(s["ctx"], s["p"].layers, s["p"].reg, s["p"].ws)
        return s
    s["p"] = _Params(s["ctx"], net, gen, W.choose_kept(net, counts, seed))
    s["new"] = _Params(s["ctx"], pruned)
    s["new2old"] = torch.full((sum(net.space_sizes),), -1, dtype=torch.int32, device="cuda")
    return s


def prepare(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "conv":
        s = _conv_state(case, gen)
    elif kind == "layer":
        s = _layer_state(case, gen)
    elif kind == "step":
        s = _step_state(case, seed)
    elif kind in ("lasso", "reconfigure"):
        s = _model_state(case, gen, seed)
    else:
        N, H, C, S = (case[k] for k in ("N", "H", "C", "S"))
        s = dict(ctx=B.Context(0), npix=N * H * H, ld=W.pad8(C), lds=W.pad8(S))
        s["idx"] = torch.sort(torch.randperm(C, generator=gen, device="cuda")[:S])[0].to(torch.int32)
        s["node"] = _act(gen, N, H, H, s["ld"])
        s["back"] = _grad(gen, N, H, H, s["lds"])
        s["branch"], s["out"] = torch.zeros_like(s["back"]), torch.zeros_like(s["node"])
    s["case"] = case
    return s


# ------------------------------------------------------------------------------------------------ run
def _run_conv(s):
    c, d = s["ctx"], s["d"]
    B.pt_conv_fwd(c, d, s["x"], s["w"], s["y"], s["ws"])
    if s["case"]["first"]:
        B.pt_conv_wgrad(c, d, s["x"], s["dy"], s["dw"], s["ws"])
        return s["y"], s["dw"]
    B.pt_conv_dgrad(c, d, s["dy"], s["w"], s["dx"], s["ws"])
    B.pt_conv_wgrad(c, d, s["x"], s["dy"], s["dw"], s["ws"])
    return s["y"], s["dx"], s["dw"]


def _run_layer(s):
    c, d, bn = s["ctx"], s["d"], s["bn"]
    parts = B.pt_conv_fwd_stats(c, d, s["x"], s["w"], s["y"], s["stats"], s["ws"])
    B.pt_bn_relu_fwd_stats(c, bn, s["y"], s["res"], s["gamma"], s["beta"], s["rm"], s["rv"], s["mean"], s["invstd"], s["a"], s["stats"], parts)
    B.pt_bn_relu_bwd(c, bn, s["y0"], s["a0"], s["da"], s["gamma"], s["mean0"], s["invstd0"], s["dy"], s["dres"], s["dgamma"], s["dbeta"], s["bnws"])
    B.pt_conv_wgrad(c, d, s["x"], s["dy"], s["dw"], s["ws"])
    B.pt_conv_dgrad(c, d, s["dy"], s["w"], s["dx"], s["ws"])
    return {k: s[k] for k in ("y", "a", "mean", "invstd", "rm", "rv", "dy", "dres", "dgamma", "dbeta", "dw", "dx")}


def _run_step(s):
    ts = s["ts"]
    ts.step()
    return {"y": s["y"].all, "dx": s["dx"].all, "dw": ts.mp.g_flat, "w": ts.mp.w, "reg": ts.mp.reg, "new2old": ts.new2old}


def _run_lasso(s):
    p = s["p"]
    if s["case"]["carried"]:
        B.pt_group_lasso_sgd_step_carried(s["ctx"], p.layers, LAM, LR, MU, 0.0, p.reg, p.ws)
    else:
        B.pt_group_lasso_sgd_step(s["ctx"], p.layers, LAM, LR, MU, 0.0, p.reg, p.ws)
    return {"w": p.w.all, "v": p.v.all, "shadow": p.wb.all, "sumsq_out": p.so.all, "sumsq_in": p.si.all, "reg": p.reg}


def _run_reconfigure(s):
    c, p, n = s["ctx"], s["p"], s["new"]
    B.pt_find_zero_groups(c, p.layers, 1e-4, False, p.ws)
    sizes = B.pt_reconfigure_plan(c, p.graph, s["new2old"])
    B.pt_reconfigure(c, p.graph, s["new2old"], n.graph)
    return {"sizes": np.array(sizes), "new2old": s["new2old"], "zero_out": p.zo.all, "zero_in": p.zi.all,
            "w": n.w.all, "v": n.v.all, "shadow": n.wb.all, "bn": n.bn.all}


def _run_gate(s):
    k = s["case"]
    B.pt_channel_gather(s["ctx"], s["node"], s["ld"], k["C"], s["idx"], k["S"], s["branch"], s["lds"], s["npix"])
    B.pt_channel_scatter_add(s["ctx"], s["back"], s["lds"], s["idx"], k["S"], s["node"], s["out"], s["ld"], k["C"], s["npix"], True)
    return s["branch"], s["out"]


_RUN = {"conv": _run_conv, "layer": _run_layer, "step": _run_step, "lasso": _run_lasso, "reconfigure": _run_reconfigure, "gate": _run_gate}


def run(state):
    return _RUN[state["case"]["kind"]](state)


# ------------------------------------------------------------------------------------------------ work and tolerance
def _conv_work(N, H, C, K, R, stride, first):
    """Forward, data gradient (unless first) and weight gradient: every pass reads its two operands and writes its result."""
    P = (H + 2 * (R // 2) - R) // stride + 1
    act, w = 2.0 * N * (H * H * C + P * P * K), K * C * R * R
    passes = 2 if first else 3
    return passes * act + w * (4 + 2 * (passes - 1)), passes * 2.0 * N * P * P * K * C * R * R


def work(case):
    kind = case["kind"]
    if kind in ("conv", "layer"):
        b, f = _conv_work(case["N"], case["H"], case["C"], case["K"], case["R"], case["stride"], case.get("first", False))
        if kind == "layer":
            P = (case["H"] + 2 * (case["R"] // 2) - case["R"]) // case["stride"] + 1
            # forward: y (+ residual) in, a out; backward: y, a, da in, dy (+ dresidual) out
            b += 2.0 * case["N"] * P * P * case["K"] * (2 + 4 + (2 if case["residual"] else 0))
        return {"bytes": b, "flops": f}
    if kind == "gate":
        return {"bytes": case["N"] * case["H"] ** 2 * (4.0 * case["S"] + 4.0 * case["C"] + 2.0 * case["S"]), "flops": 0}
    net, counts, pruned = _nets(case)
    old, new = _params(net), _params(pruned)
    lasso = new * 22.0                               # w, g, v in; w, v, shadow out
    move = old * 4.0 + new * 18.0                    # detection reads w; the gather reads w, v and writes w, v, shadow
    if kind == "lasso":
        return {"bytes": lasso, "flops": 12.0 * new}
    if kind == "reconfigure":
        return {"bytes": move, "flops": 0}
    both = [_conv_work(case["N"], l.H, l.C, l.K, l.R, l.stride, i == 0) for i, l in enumerate(pruned.layers)]
    return {"bytes": lasso + move + sum(b for b, _ in both), "flops": sum(f for _, f in both)}


def tolerance(case):
    kind = case["kind"]
    if kind in ("reconfigure", "gate"):
        return "exact"                               # data movement, and one rounding of a sum of two values
    if kind == "lasso":
        return {"rel": 1e-4, "max": 1e-2}            # 32-bit sums; the bf16 shadow may round the other way
    return {"rel": 5e-3, "max": 2e-2}                # bf16 results of 32-bit accumulation
