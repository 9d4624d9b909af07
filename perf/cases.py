"""The layer calls whose speed is measured: what a program that uses this
framework asks of it, from one small fp32 batch to the largest training step.

Kinds of case (``kind``):

* ``step``     one forward + backward of ``MoeLayer``, eager or (``graph``) the
               replay of its captured CUDA graph, as a training loop runs it;
* ``forward``  ``MoeLayer.forward`` alone, as evaluation and serving run it;
* ``experts``  the expert FFN block, forward and backward, on given rows
               (``moe_expert_ffn``, ``moe_expert_ffn_bwd``), for a caller that
               does its own routing;
* ``route``    the router alone: logits, top-K and probabilities
               (``moe_route``);
* ``payload``  dispatch through a low-precision payload and its arrival
               (``moe_dispatch_fp8`` / ``moe_dequant_rows``,
               ``moe_dispatch_nvfp4`` / ``moe_dequant_nvfp4``).

Inputs are N(0, 1) activations and upstream gradients and weights of variance
1 / fan_in, drawn on the GPU from the seed; ``skew`` adds the logit bias
3 ln(1 / (e + 1)), which sends most slots to the first experts and leaves many
without rows.
"""
from __future__ import annotations

import math

import torch

from paper_2608_28511_gb300 import abi
from paper_2608_28511_gb300.layer import MoeLayer


def _case(name, kind, **kw):
    c = {"kind": kind, "S": 1, "GBS": 1, "K": 1, "D": 64, "E": 1, "F": 64, "H": 0, "dtype": "bf16",
         "router": "softmax", "shared_F": 0, "payload": "bf16", "skew": False, "graph": False}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest step: an fp32 layer of a unit test or a debugging run,
        # where launches and latency are all there is
        _case("step_fp32_T256", "step", S=128, GBS=2, K=2, D=128, E=8, F=256, dtype="f32", graph=True),
        # an fp32 reference run of a mid-sized layer, odd token and expert counts
        _case("step_fp32_T3001", "step", S=3001, GBS=1, K=3, D=512, E=12, F=768, dtype="f32"),
        # evaluation of a few tokens: every expert's weights are read for a row or two each
        _case("forward_T64", "forward", S=64, GBS=1, K=6, D=2048, E=64, F=1024),
        # evaluation of one odd-sized batch with the wider experts
        _case("forward_T1999", "forward", S=1999, GBS=1, K=8, D=2048, E=128, F=1536),
        # a small training micro-batch; the number of experts is not a multiple of 8
        _case("step_T2045_E60", "step", S=2045, GBS=1, K=4, D=2048, E=60, F=1408),
        # the base training step
        _case("step_base", "step", S=4096, GBS=2, K=6, D=2048, E=64, F=1024, graph=True),
        # the largest training step, skewed routing
        _case("step_skew", "step", S=8192, GBS=4, K=8, D=2048, E=128, F=1024, skew=True, graph=True),
        # LatentMoE: model width 4096 projected down to 1024 before the dispatch
        _case("step_latent", "step", S=4096, GBS=4, K=8, D=1024, E=256, F=768, H=4096, graph=True),
        # the router and shared expert of the paper's own runs
        _case("step_sigmoid_shared", "step", S=4096, GBS=2, K=6, D=2048, E=64, F=1024, router="sigmoid",
              shared_F=2688, graph=True),
        # the expert block on ragged groups and widths that are not whole tiles
        _case("experts_T8191", "experts", S=8191, GBS=1, K=4, D=1408, E=60, F=704),
        # the router of an odd-sized large batch
        _case("route_T30011", "route", S=30011, GBS=1, K=8, D=2048, E=128),
        # an NVFP4 dispatch and its arrival
        _case("payload_nvfp4_T8191", "payload", S=8191, GBS=1, K=6, D=2048, E=64, payload="nvfp4"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _m64(rng, lo, hi):
    return max(lo // 64, min(hi // 64, int(round(_log(rng, lo, hi) / 64)))) * 64


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "step_f32", "forward", "forward", "experts", "route",
                       "payload"])
    if kind == "step_f32":
        E = rng.randint(4, 32)
        return _case(None, "step", S=_log(rng, 64, 3001), K=rng.randint(1, 4), D=_m64(rng, 64, 512), E=E,
                     F=_m64(rng, 64, 768), dtype="f32", graph=rng.random() < 0.5)
    D, F = _m64(rng, 256, 2560), _m64(rng, 128, 1536)
    E = rng.choice([8 * rng.randint(1, 16), 4 * rng.randint(2, 32), rng.choice([160, 192, 256])])
    K = rng.randint(1, min(8, E))
    # no more rows, expert weights or arithmetic than the largest listed step
    E = min(E, max(8, 128 * 2048 * 1024 // (D * F) // 8 * 8))
    K = min(K, E)
    T = min(_log(rng, 16, 32768), 262144 // K, int(262144 * 2048 * 1024 / (K * D * F)))
    if kind == "route":
        return _case(None, "route", S=_log(rng, 64, 32768), K=K, D=_m64(rng, 512, 4096), E=E,
                     skew=rng.random() < 0.3)
    if kind == "payload":
        return _case(None, "payload", S=_log(rng, 64, 16384), K=K, D=D, E=E, payload=rng.choice(["fp8", "nvfp4"]))
    if kind == "experts":
        return _case(None, "experts", S=min(T, 16384), K=K, D=D, E=E, F=F, skew=rng.random() < 0.3)
    router = rng.choice(["softmax", "softmax", "sigmoid"])
    H = 0
    if rng.random() < 0.25:
        D = _m64(rng, 256, 1024)
        H = D * rng.choice([2, 4])
    shared = _m64(rng, 256, 2688) if rng.random() < 0.25 else 0
    if H or shared:
        T = min(T, 16384)
    GBS = rng.choice([1, 1, 2]) if T > 1 else 1
    return _case(None, kind, S=T // GBS, GBS=GBS, K=K, D=D, E=E, F=F, H=H,
                 router=router, shared_F=shared, payload=rng.choice(["bf16", "bf16", "bf16", "fp8", "nvfp4"]),
                 skew=router == "softmax" and rng.random() < 0.3, graph=kind == "step" and rng.random() < 0.5)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
_AUX_COEF, _AUX_GRAD = 1e-4, 1.0


def _dt(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def _skew_bias(E):
    return torch.tensor([3.0 * math.log(1.0 / (e + 1)) for e in range(E)], dtype=torch.float32, device="cuda")


def _inputs(c, seed):
    """The case's inputs on the GPU, from the seed alone."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    dt = _dt(c)
    T, K, D, E, F, H, Fs = c["S"] * c["GBS"], c["K"], c["D"], c["E"], c["F"], c["H"], c["shared_F"]
    X = H or D

    def randn(*shape, std=1.0, dtype=dt):
        return (torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32) * std).to(dtype)

    bias = _skew_bias(E) if c["skew"] else None
    if c["kind"] == "route":
        return {"x": randn(T, D), "w_router": randn(E, D, std=D ** -0.5), "bias": bias}
    if c["kind"] in ("experts", "payload"):
        z = randn(T, E, dtype=torch.float32)
        z = z if bias is None else z + bias
        top = torch.topk(z, K, dim=1)
        idx, prob = top.indices.to(torch.int32).contiguous(), torch.softmax(top.values, dim=1).contiguous()
        if c["kind"] == "payload":
            return {"x": randn(T, D), "idx": idx, "prob": prob}
        off = torch.zeros(E + 1, dtype=torch.int32, device="cuda")
        off[1:] = torch.cumsum(torch.bincount(idx.reshape(-1).long(), minlength=E), 0).to(torch.int32)
        return {"x_perm": randn(T * K, D), "offsets": off, "w_gate": randn(E, F, D, std=D ** -0.5),
                "w_up": randn(E, F, D, std=D ** -0.5), "w2": randn(E, D, F, std=F ** -0.5),
                "dy_perm": randn(T * K, D, std=1.0 / K)}
    d = {"x": randn(T, X), "w_router": randn(E, X, std=X ** -0.5), "w_gate": randn(E, F, D, std=D ** -0.5),
         "w_up": randn(E, F, D, std=D ** -0.5), "w2": randn(E, D, F, std=F ** -0.5), "dy": randn(T, X), "bias": bias}
    if H:
        d["w_down"], d["w_upp"] = randn(D, H, std=H ** -0.5), randn(H, D, std=D ** -0.5)
    if Fs:
        d["w_s1"], d["w_s2"] = randn(Fs, X, std=X ** -0.5), randn(X, Fs, std=Fs ** -0.5)
    if c["router"] == "sigmoid":
        d["expert_bias"] = randn(E, std=0.05, dtype=torch.float32)
    return d


def prepare(case, seed):
    c = case
    d = _inputs(c, seed)
    T, K, D, E, F = c["S"] * c["GBS"], c["K"], c["D"], c["E"], c["F"]
    dt = _dt(c)

    def empty(*shape, dtype=dt):
        return torch.empty(*shape, dtype=dtype, device="cuda")

    if c["kind"] in ("step", "forward"):
        layer = MoeLayer(c["S"], c["GBS"], K, D, E, F, c["dtype"], c["H"], router=c["router"], aux_coef=_AUX_COEF,
                         aux_grad=_AUX_GRAD, shared_F=c["shared_F"], payload=c["payload"])
        layer.load(d)
        st = {"kind": c["kind"], "layer": layer, "graph": None}
        if c["graph"]:
            layer.step()
            st["graph"] = layer.capture()
        return st
    shape = abi.MoeShape.of(c["S"], c["GBS"], K, D, E, F, c["dtype"])
    st = {"kind": c["kind"], "shape": shape,
          "ws": torch.empty(abi.moe_workspace_size(shape), dtype=torch.uint8, device="cuda")}
    st.update(d)
    f32, i32, u8 = torch.float32, torch.int32, torch.uint8
    if c["kind"] == "route":
        st.update(logits=empty(T, E, dtype=f32), idx=empty(T, K, dtype=i32), prob=empty(T, K, dtype=f32))
    elif c["kind"] == "experts":
        st["w1"] = empty(E, 2 * F, D)
        abi.moe_pack_w1(shape, st.pop("w_gate"), st.pop("w_up"), st["w1"])
        st.update(h=empty(T * K, 2 * F), act=empty(T * K, F), y_perm=empty(T * K, D), dx_perm=empty(T * K, D),
                  dw1=empty(E, 2 * F, D, dtype=f32), dw2=empty(E, D, F, dtype=f32))
    else:
        st.update(payload=c["payload"], offsets=empty(E + 1, dtype=i32), row_of_slot=empty(T * K, dtype=i32),
                  token_of_row=empty(T * K, dtype=i32), prob_perm=empty(T * K, dtype=f32), x_perm=empty(T * K, D),
                  codes=empty(T * K, D if c["payload"] == "fp8" else D // 2, dtype=u8),
                  bscale=empty(T * K, D // 16, dtype=u8), rscale=empty(T * K, dtype=f32))
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(state):
    s = state
    if s["kind"] in ("step", "forward"):
        L = s["layer"]
        if s["kind"] == "forward":
            L.forward()
        elif s["graph"] is not None:
            s["graph"].replay()
        else:
            L.step()
        out = {"y": L.y, "logits": L.logits, "topk_idx": L.topk_idx, "topk_prob": L.topk_prob}
        if L.router == "sigmoid":
            out["aux_loss"] = L.aux_loss[:1]
        if s["kind"] == "step":
            out.update(dx=L.dx, dw1=L.dw1, dw2=L.dw2, dw_router=L.dw_router)
            if L.H:
                out.update(dw_down=L.dw_down, dw_upp=L.dw_upp)
            if L.shared_F:
                out.update(dw_s1=L.dw_s1, dw_s2=L.dw_s2)
        return out
    if s["kind"] == "route":
        abi.moe_route(s["shape"], s["x"], s["w_router"], s["bias"], s["logits"], s["idx"], s["prob"], s["ws"])
        return {"logits": s["logits"], "topk_idx": s["idx"], "topk_prob": s["prob"]}
    if s["kind"] == "experts":
        abi.moe_expert_ffn(s["shape"], s["x_perm"], s["offsets"], s["w1"], s["w2"], s["h"], s["act"], s["y_perm"],
                           s["ws"])
        abi.moe_expert_ffn_bwd(s["shape"], s["dy_perm"], s["x_perm"], s["h"], s["act"], s["offsets"], s["w1"],
                               s["w2"], s["dx_perm"], s["dw1"], s["dw2"], s["ws"])
        return {k: s[k] for k in ("h", "act", "y_perm", "dx_perm", "dw1", "dw2")}
    common = (s["shape"], s["x"], s["idx"], s["prob"], s["offsets"], s["row_of_slot"], s["token_of_row"], s["codes"])
    names = ["offsets", "row_of_slot", "token_of_row", "prob_perm", "codes", "rscale", "x_perm"]
    if s["payload"] == "fp8":
        abi.moe_dispatch_fp8(*common, s["rscale"], s["prob_perm"], s["ws"])
        abi.moe_dequant_rows(s["shape"], s["codes"], s["rscale"], s["x_perm"])
    else:
        abi.moe_dispatch_nvfp4(*common, s["bscale"], s["rscale"], s["prob_perm"], s["ws"])
        abi.moe_dequant_nvfp4(s["shape"], s["codes"], s["bscale"], s["rscale"], s["x_perm"])
        names.append("bscale")
    return {k: s[k] for k in names}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    c = case
    T, K, D, E, F, H, Fs = c["S"] * c["GBS"], c["K"], c["D"], c["E"], c["F"], c["H"], c["shared_F"]
    TK, X, b = T * K, H or D, 2 if c["dtype"] == "bf16" else 4
    # experts that get rows: all of those that T K slots can reach, about a
    # quarter of them under the skewed bias; the others' weights need no reading
    reached = min(E, TK) if not c["skew"] else min(max(K, E // 4), TK)
    weights = 3 * reached * D * F * b
    route = {"bytes": T * X * b + E * X * b + 4 * T * E + 8 * TK, "flops": 2.0 * T * X * E}
    if c["kind"] == "route":
        return route
    if c["kind"] == "payload":
        q = D if c["payload"] == "fp8" else D // 2 + D // 16
        return {"bytes": T * D * 2 + 8 * TK + TK * (q + 4) + TK * (D * 2 + 12), "flops": 0.0}
    if c["kind"] == "experts":
        return {"bytes": 2 * weights + TK * (2 * D + 3 * F + 2 * D) * b + 3 * E * D * F * 4,
                "flops": 18.0 * TK * D * F}
    dense = 2 * H * D + 2 * Fs * X
    out = {"bytes": route["bytes"] + T * X * b + weights + dense * b,
           "flops": route["flops"] + 6.0 * TK * D * F + 2.0 * T * dense}
    if c["kind"] == "step":
        # dy in, dx out; the weights again for the input gradients; fp32 weight gradients
        out["bytes"] += 2 * T * X * b + weights + dense * b + 4 * (3 * E * D * F + E * X + dense)
        out["flops"] *= 3
    return out


def tolerance(case):
    c = case
    if c["kind"] == "payload":
        return "exact"
    if c["kind"] == "route":
        # fp32 sums of D products; two equal or nearly equal logits may change places
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    if c["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    if c["kind"] == "experts":
        return {"rel": 1e-2}
    # bf16 activations between the stages.  Logits within an fp32 rounding of
    # each other may pick another K-th expert for a token, whose y and dx then
    # change by up to about their own root mean square: "max" allows that,
    # "rel" only a few such tokens.
    return {"rel": 1e-2, "max": 0.9, "differ": 1e-3}


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _pack(g, u):
    """[..., F, D] gate and up rows in the packed order: blocks of 64 gate rows, then their 64 up rows."""
    F, D = g.shape
    return torch.stack([g.view(F // 64, 64, D), u.view(F // 64, 64, D)], 1).reshape(2 * F, D)


def _expert(xe, wg, wu, w2, dye=None):
    """One expert's SwiGLU FFN on rows xe and, given the gradient of its output, the backward."""
    g, u = xe @ wg.T, xe @ wu.T
    s = torch.sigmoid(g)
    a = g * s * u
    y = a @ w2.T
    if dye is None:
        return g, u, a, y
    da = dye @ w2
    dg, du = da * u * s * (1 + g * (1 - s)), da * g * s
    return g, u, a, y, dg @ wg + du @ wu, dg.T @ xe, du.T @ xe, dye.T @ a


def exact(case, seed):
    c = case
    if work(c)["flops"] > 1.2e13:
        return None  # over about 20 seconds of 64-bit arithmetic
    d = _inputs(c, seed)
    T, K, D, E, F, H, Fs = c["S"] * c["GBS"], c["K"], c["D"], c["E"], c["F"], c["H"], c["shared_F"]
    f64 = torch.float64

    def zeros(*shape):
        return torch.zeros(*shape, dtype=f64, device="cuda")

    if c["kind"] == "payload":
        # the probabilities travel unchanged, in a stable order by expert; codes
        # and scales are defined by their own roundings
        order = torch.sort(d["idx"].reshape(-1).long(), stable=True).indices
        return {"prob_perm": d["prob"].reshape(-1)[order].double(), "codes": None, "x_perm": None, "rscale": None}
    if c["kind"] == "experts":
        off = d["offsets"].tolist()
        TK = T * K
        o = {"h": zeros(TK, 2 * F), "act": zeros(TK, F), "y_perm": zeros(TK, D), "dx_perm": zeros(TK, D),
             "dw1": torch.zeros(E, 2 * F, D, device="cuda"), "dw2": torch.zeros(E, D, F, device="cuda")}
        for e in range(E):
            r = slice(off[e], off[e + 1])
            if r.start == r.stop:
                continue
            g, u, a, y, dx, dwg, dwu, dw2 = _expert(d["x_perm"][r].to(f64), d["w_gate"][e].to(f64),
                                                    d["w_up"][e].to(f64), d["w2"][e].to(f64),
                                                    d["dy_perm"][r].to(f64))
            o["h"][r] = _pack(g.T, u.T).T
            o["act"][r], o["y_perm"][r], o["dx_perm"][r] = a, y, dx
            o["dw1"][e], o["dw2"][e] = _pack(dwg, dwu).float(), dw2.float()
        return o
    x = d["x"].to(f64)
    wr = d["w_router"].to(f64)
    z = x @ wr.T
    if d["bias"] is not None:
        z = z + d["bias"].to(f64)
    if c["router"] == "sigmoid":
        sc = torch.sigmoid(z)
        idx = torch.topk(sc + d["expert_bias"].to(f64), K, dim=1).indices
        sel = sc.gather(1, idx)
        prob = sel / sel.sum(1, keepdim=True)
    else:
        top = torch.topk(z, K, dim=1)
        idx, prob = top.indices, torch.softmax(top.values, dim=1)
    out = {"logits": z, "topk_idx": None, "topk_prob": prob}
    if c["kind"] == "route":
        return out
    step = c["kind"] == "step"
    xd = x @ d["w_down"].to(f64).T if H else x
    if c["payload"] != "bf16":
        return out  # the payload's own roundings are not part of a 64-bit result
    y = zeros(T, D)
    dy = d["dy"].to(f64) if step else None
    dyd = (dy @ d["w_upp"].to(f64) if H else dy) if step else None
    dprob, dxd = zeros(T, K), zeros(T, D)
    if step:
        out["dw1"], out["dw2"] = torch.zeros(E, 2 * F, D, device="cuda"), torch.zeros(E, D, F, device="cuda")
    for e in range(E):
        t, k = torch.nonzero(idx == e, as_tuple=True)
        if not t.numel():
            continue
        w = d["w_gate"][e].to(f64), d["w_up"][e].to(f64), d["w2"][e].to(f64)
        p = prob[t, k].unsqueeze(1)
        if not step:
            y.index_add_(0, t, p * _expert(xd[t], *w)[3])
            continue
        dyt = dyd[t]
        g, u, a, ye, dx, dwg, dwu, dw2 = _expert(xd[t], *w, p * dyt)
        y.index_add_(0, t, p * ye)
        dprob[t, k] = (dyt * ye).sum(1)
        dxd.index_add_(0, t, dx)
        out["dw1"][e], out["dw2"][e] = _pack(dwg, dwu).float(), dw2.float()
    out["y"] = y @ d["w_upp"].to(f64).T if H else y
    if Fs:
        h = x @ d["w_s1"].to(f64).T
        act = torch.relu(h) ** 2
        out["y"] = out["y"] + act @ d["w_s2"].to(f64).T
    if c["router"] == "sigmoid":
        S, G = c["S"], c["GBS"]
        f = zeros(T, E).scatter_(1, idx, 1.0).view(G, S, E).sum(1) * (E / (K * S))
        tot = sc.sum(1, keepdim=True)
        P = (sc / tot).view(G, S, E).mean(1)
        out["aux_loss"] = (_AUX_COEF / G * (f * P).sum()).reshape(1)
    if not step:
        return out
    dot = (prob * dprob).sum(1, keepdim=True)
    if c["router"] == "sigmoid":
        ds = zeros(T, E).scatter_(1, idx, (dprob - dot) / sel.sum(1, keepdim=True))
        cg = (_AUX_GRAD * _AUX_COEF / (G * S) * f).repeat_interleave(S, 0)
        ds += (cg - (cg * sc / tot).sum(1, keepdim=True)) / tot
        dz = sc * (1 - sc) * ds
    else:
        dz = zeros(T, E).scatter_(1, idx, prob * (dprob - dot))
    out["dw_router"] = dz.T @ x
    dx = dz @ wr
    if H:
        dx += dxd @ d["w_down"].to(f64)
        out["dw_down"], out["dw_upp"] = dxd.T @ x, dy.T @ y
    else:
        dx += dxd
    if Fs:
        dh = 2 * torch.relu(h) * (dy @ d["w_s2"].to(f64))
        dx += dh @ d["w_s1"].to(f64)
        out["dw_s1"], out["dw_s2"] = dh.T @ x, dy.T @ act
    out["dx"] = dx
    return out
