"""Timed cases of the MoE expert layer: what a training program has the library do.

Whole layer calls (paper_2601_14327_gb300.layer: forward, and forward + backward) and
the entry points a program with a layer of its own calls one by one (the C ABI through
paper_2601_14327_gb300._lib), from a forward over a few dozen tokens to the largest
single-GPU layer. Inputs are synthetic and seeded, with the distributions of the
package's own workloads: x, dy ~ N(0,1) in bf16, expert weights ~ N(0, 0.02) in bf16, an fp32
router ~ N(0, 1/d) with a fixed gate bias that sets the load skew.

A case is a dict: kind (what is called), T tokens, d = d_model, E experts, k experts per
token, F = d_ff, bias ("none", "zipf", "loguniform"), zipf_s, pruned (experts masked out).
"""
import math

import torch

from paper_2601_14327_gb300 import _lib as L
from paper_2601_14327_gb300 import layer

PAD = 128      # rows of a group are padded to this
BF16, F32, F64, I32 = torch.bfloat16, torch.float32, torch.float64, torch.int32


def _case(name, kind, T, d, E, k, F=0, bias="none", zipf_s=1.2, pruned=0):
    c = {"kind": kind, "T": T, "d": d, "E": E, "k": k, "F": F, "bias": bias, "zipf_s": zipf_s,
         "pruned": pruned}
    return {"name": name, **c} if name else c


def listed():
    return [
        # ---- whole layer calls
        # a validation pass over a short ragged sequence through a trained, skewed layer:
        # almost every expert gets a row or two, so the weights are what is read
        _case("fwd_few_tokens", "layer_fwd", 37, 2048, 64, 6, 1408, "zipf"),
        # the smallest configuration: launches and latency count
        _case("fwd_tiny", "layer_fwd", 512, 256, 16, 2, 512),
        # steady but imbalanced load, forward only
        _case("fwd_skew", "layer_fwd", 8192, 2048, 64, 6, 1408, "zipf"),
        # a training step of a small model on a ragged token count, d_ff not a multiple of 256
        _case("step_small", "layer_step", 1021, 512, 32, 4, 384, "zipf"),
        # a training step with 16 of 64 experts pruned by mask
        _case("step_pruned", "layer_step", 16384, 4096, 64, 8, 2048, "zipf", pruned=16),
        # the largest layer: 256 experts of which 171 are left after pruning
        _case("step_large", "layer_step", 65536, 7168, 171, 8, 2048, "zipf", 1.0),
        # ---- entry points one by one
        # the router of the 128-expert layer under volatile load (some experts get nothing)
        _case("route_volatile", "route", 32768, 4096, 128, 8, bias="loguniform"),
        # the router's backward on a ragged micro-batch of the wide model
        _case("route_bwd_ragged", "route_bwd", 8191, 7168, 171, 8, bias="zipf", zipf_s=1.0),
        # recording the load statistic and grouping the tokens, pruned layer
        _case("dispatch_pruned", "dispatch", 16384, 4096, 64, 8, bias="zipf", pruned=16),
        # back to token order: a micro-batch of ragged length
        _case("combine_ragged", "combine", 4093, 2048, 64, 6, bias="zipf"),
        # the experts' FFN alone on a micro-batch, volatile load
        _case("ffn_fwd_volatile", "ffn_fwd", 4096, 4096, 128, 8, 1536, "loguniform"),
        # its backward, on a small ragged one
        _case("ffn_bwd_ragged", "ffn_bwd", 2039, 2048, 64, 6, 1408, "zipf"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges, sizes spread over their logarithms."""
    kinds = ("layer_fwd", "layer_fwd", "layer_step", "layer_step", "route", "route_bwd",
             "dispatch", "combine", "ffn_fwd", "ffn_bwd")
    top = listed()[5]
    while True:
        kind = rng.choice(kinds)
        step = 128 if kind.startswith(("layer", "ffn")) else 8
        E = _log_int(rng, 8, 256)
        c = _case("", kind, _log_int(rng, 32, 65536), step * _log_int(rng, 256 // step, 7168 // step),
                  E, rng.randint(1, min(8, E)),
                  128 * _log_int(rng, 2, 16) if step == 128 else 0,
                  rng.choice(("none", "zipf", "zipf", "loguniform")), rng.choice((0.8, 1.0, 1.2)))
        if kind.startswith("layer") or kind == "dispatch":
            c["pruned"] = rng.choice((0, 0, (E - c["k"]) // 4))
        if _state_bytes(c) <= _state_bytes(top) and work(c)["flops"] <= work(top)["flops"]:
            return c


# ---------------------------------------------------------------- inputs


def _rows_cap(c):
    return c["T"] * c["k"] + PAD * c["E"]


def _state_bytes(c):
    """Device memory of a prepared case, about."""
    T, d, E, F, R = c["T"], c["d"], c["E"], c["F"], _rows_cap(c)
    if c["kind"] == "layer_step":
        return 2 * (4 * R * d + 6 * R * F + 6 * E * d * F + 6 * T * d) + 40 * T * E
    return 2 * (2 * R * d + 3 * R * F + 3 * E * d * F + 3 * T * d) + 40 * T * E


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(1000 + int(seed))


def _randn(g, *shape, std=1.0, dtype=BF16):
    return torch.empty(*shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=g)


def _bias_and_mask(c, g):
    """The fixed gate bias, and the mask of the experts that pruning left (None: all)."""
    E = c["E"]
    if c["bias"] == "zipf":
        bias = -c["zipf_s"] * torch.log(1.0 + torch.randperm(E, generator=g, device="cuda").double())
    elif c["bias"] == "loguniform":
        bias = 7.0 * torch.rand(E, generator=g, device="cuda", dtype=F64) - 7.0
        bias[torch.argsort(bias)[:min(8, E // 4, E - c["k"])]] = -30.0
    else:
        bias = torch.zeros(E, device="cuda", dtype=F64)
    mask = None
    if c["pruned"]:  # the experts that the bias gives the least load
        order = torch.argsort(bias, stable=True)
        mask = torch.ones(E, dtype=torch.uint8, device="cuda")
        mask[order[:c["pruned"]]] = 0
    return bias.float(), mask


def _weights(c, g):
    E, d, F = c["E"], c["d"], c["F"]
    return _randn(g, E, 2 * F, d, std=0.02), _randn(g, E, d, F, std=0.02)


def _router(c, g):
    return _randn(g, c["d"], c["E"], std=1.0 / math.sqrt(c["d"]), dtype=F32)


def _routing(c, g):
    """A routing as the router leaves it: topk_idx, topk_gate, the mask of its experts."""
    bias, mask = _bias_and_mask(c, g)
    z = _randn(g, c["T"], c["E"], dtype=F32) + bias
    if mask is not None:
        z[:, mask == 0] = -math.inf
    v, idx = torch.topk(z, c["k"], dim=1)
    return idx.to(I32).contiguous(), torch.softmax(v, dim=1).contiguous(), mask


def _layout(idx, E):
    """Grouped layout of a routing: group_offsets, group_counts, row_of_assignment."""
    flat = idx.reshape(-1).long()
    counts = torch.bincount(flat, minlength=E)
    padded = (counts + PAD - 1) // PAD * PAD
    off = torch.zeros(E + 1, dtype=torch.long, device=flat.device)
    off[1:] = torch.cumsum(padded, 0)
    first = torch.cumsum(counts, 0) - counts
    order = torch.argsort(flat, stable=True)
    row = torch.empty_like(flat)
    e = flat[order]
    row[order] = off[e] + torch.arange(flat.numel(), device=flat.device) - first[e]
    return off.to(I32), counts.to(I32), row.reshape(idx.shape).to(I32)


def _grouped(c, rows, row, scale=None):
    """[R, d] with rows[t] (times scale[t, j]) at the row of every assignment, zeros elsewhere."""
    out = torch.zeros(_rows_cap(c), rows.shape[1], dtype=rows.dtype, device=rows.device)
    for j in range(c["k"]):
        v = rows if scale is None else (rows.float() * scale[:, j:j + 1]).to(rows.dtype)
        out[row[:, j].long()] = v
    return out


def _block(m):
    """[R, 2F] row-major -> the 32-row blocked layout of the saved pre-activations (the rows
    past the last whole block belong to no group)."""
    out, C = torch.zeros_like(m), m.shape[1]
    n = m.shape[0] // 32 * 32
    out[:n] = m[:n].reshape(n // 32, 32, C // 8, 8).transpose(1, 2).reshape(n, C)
    return out


def _inputs(c, seed):
    """The case's inputs, a function of the seed alone."""
    g, T, d, E, k, F = _generator(seed), c["T"], c["d"], c["E"], c["k"], c["F"]
    kind, s = c["kind"], {}
    if kind.startswith("layer") or kind == "route":
        s["bias"], s["mask"] = _bias_and_mask(c, g)
        s["x"], s["w_router"] = _randn(g, T, d), _router(c, g)
        if kind != "route":
            s["w_gate_up"], s["w_down"] = _weights(c, g)
        if kind == "layer_step":
            s["dy"] = _randn(g, T, d)
        return s
    s["idx"], s["gate"], s["mask"] = _routing(c, g)
    if kind == "route_bwd":
        s["x"], s["d_gate"] = _randn(g, T, d), _randn(g, T, k, dtype=F32)
        return s
    if kind == "dispatch":
        s["x"] = _randn(g, T, d)
        return s
    s["off"], s["count"], s["row"] = _layout(s["idx"], E)
    if kind == "combine":
        s["out_perm"] = torch.zeros(_rows_cap(c), d, dtype=BF16, device="cuda")
        for j in range(k):
            s["out_perm"][s["row"][:, j].long()] = _randn(g, T, d)
        return s
    s["w_gate_up"], s["w_down"] = _weights(c, g)
    s["x_perm"] = _grouped(c, _randn(g, T, d), s["row"])
    if kind == "ffn_bwd":
        R, std = _rows_cap(c), 0.02 * math.sqrt(d)
        live = torch.zeros(R, 1, dtype=BF16, device="cuda")
        live[s["row"].reshape(-1).long()] = 1
        s["ab"] = _randn(g, R, 2 * F, std=std) * live     # row-major; prepare() blocks it
        a, b = s["ab"][:, :F].float(), s["ab"][:, F:].float()
        s["h"] = (a * torch.sigmoid(a) * b).to(BF16)
        s["d_out"] = _grouped(c, _randn(g, T, d), s["row"], s["gate"])
        s["w_router"] = _router(c, g)
    return s


def prepare(case, seed):
    c, s = case, _inputs(case, seed)
    T, d, E, k, F, R = c["T"], c["d"], c["E"], c["k"], c["F"], _rows_cap(case)
    s["case"], kind = c, case["kind"]

    def zeros(*shape, dtype=BF16):
        return torch.zeros(*shape, dtype=dtype, device="cuda")

    if kind.startswith("layer"):
        s["buf"] = layer.MoELayerBuffers(layer.LayerShape(T, d, E, k, F), "cuda",
                                         backward=kind == "layer_step")
        if kind == "layer_step":  # pruned experts' gradients are not written
            s["buf"].dw_gate_up.zero_()
            s["buf"].dw_down.zero_()
        return s
    s["ws_bytes"] = max(L.moe_workspace_size(T, d, E, k, max(F, 128)), 256)
    s["ws"] = torch.empty(s["ws_bytes"], dtype=torch.uint8, device="cuda")
    if kind == "route":
        s["idx"], s["gate"] = zeros(T, k, dtype=I32), zeros(T, k, dtype=F32)
        s["counts"] = zeros(E, dtype=I32)
    elif kind == "route_bwd":
        s["d_logits"], s["dw_router"] = zeros(T, k, dtype=F32), zeros(d, E, dtype=F32)
    elif kind == "dispatch":
        s["counts"], s["off"] = zeros(E, dtype=I32), zeros(E + 1, dtype=I32)
        s["count"], s["row"] = zeros(E, dtype=I32), zeros(T, k, dtype=I32)
        s["x_perm"] = zeros(R, d)
    elif kind == "combine":
        s["y"] = zeros(T, d)
    elif kind == "ffn_fwd":
        s["ab"], s["h"], s["out_perm"] = zeros(R, 2 * F), zeros(R, F), zeros(R, d)
    else:
        s["ab"] = _block(s["ab"])
        s["d_gate"], s["d_ab"], s["dx_perm"] = zeros(T, k, dtype=F32), zeros(R, 2 * F), zeros(R, d)
        s["dw_gate_up"], s["dw_down"] = zeros(E, 2 * F, d), zeros(E, d, F)
    return s


def run(s):
    c = s["case"]
    T, d, E, k, F, R, kind = c["T"], c["d"], c["E"], c["k"], c["F"], _rows_cap(c), c["kind"]
    if kind.startswith("layer"):
        b = s["buf"]
        y = layer.forward(b, s["x"], s["w_router"], s["bias"], s["w_gate_up"], s["w_down"], s["mask"])
        out = {"y": y, "idx": b.topk_idx, "gate": b.topk_gate}
        if kind == "layer_step":
            dx, dgu, ddn, dr = layer.backward(b, s["dy"], s["w_router"], s["w_gate_up"], s["w_down"],
                                              active_mask=s["mask"])
            out.update(dx=dx, dw_gate_up=dgu, dw_down=ddn, dw_router=dr)
        return out
    if kind == "route":
        # (the counts are the histogram of idx, which is returned whole)
        L.moe_route(s["x"], s["w_router"], s["bias"], s["mask"], T, d, E, k, None, None, s["idx"],
                    s["gate"], s["counts"], s["ws"], s["ws_bytes"])
        return {"idx": s["idx"], "gate": s["gate"]}
    if kind == "route_bwd":
        L.moe_route_bwd(s["x"], s["idx"], s["gate"], s["d_gate"], T, d, E, k, s["d_logits"],
                        s["dw_router"], s["ws"], s["ws_bytes"])
        return {"d_logits": s["d_logits"], "dw_router": s["dw_router"]}
    if kind == "dispatch":
        L.moe_load_stats(s["idx"], T, k, E, s["counts"])
        L.moe_permute(s["x"], s["idx"], s["counts"], T, d, E, k, R, s["off"], s["count"], s["row"],
                      s["x_perm"], s["ws"], s["ws_bytes"])
        return {"counts": s["counts"], "off": s["off"], "count": s["count"], "row": s["row"],
                "x_perm": s["x_perm"]}
    if kind == "combine":
        L.moe_unpermute_combine(s["out_perm"], s["row"], s["gate"], T, d, k, s["y"])
        return {"y": s["y"]}
    if kind == "ffn_fwd":
        L.moe_grouped_ffn_fwd(s["x_perm"], s["off"], E, d, F, R, s["w_gate_up"], s["w_down"], s["ab"],
                              s["h"], s["out_perm"], s["ws"], s["ws_bytes"])
        return {"ab": s["ab"], "h": s["h"], "out": s["out_perm"]}
    L.moe_grouped_ffn_bwd(s["d_out"], s["x_perm"], s["ab"], s["h"], s["off"], s["mask"], E, d, F, R,
                          s["w_gate_up"], s["w_down"], s["gate"], None, s["row"], s["w_router"], T,
                          k, s["d_gate"], s["d_ab"], s["dx_perm"], s["dw_gate_up"], s["dw_down"],
                          s["ws"], s["ws_bytes"])
    return {"d_gate": s["d_gate"], "d_ab": s["d_ab"], "dx_perm": s["dx_perm"],
            "dw_gate_up": s["dw_gate_up"], "dw_down": s["dw_down"]}


# ---------------------------------------------------------------- what a pass needs


def work(case):
    """Bytes with every input read once and every output written once, and the operations."""
    c = case
    T, d, E, k, F = c["T"], c["d"], c["E"], c["k"], c["F"]
    A, kind = T * k, c["kind"]
    live = min(E - c["pruned"], A)                  # experts that can get a row
    weights, act, routing = 2 * 3 * live * d * F, 2 * T * d, 8 * A
    if kind == "layer_fwd":
        return {"bytes": weights + 2 * act + routing + 4 * d * E, "flops": 6 * A * d * F + 2 * T * d * E}
    if kind == "layer_step":
        return {"bytes": weights + 2 * 3 * (E - c["pruned"]) * d * F + 4 * act + routing + 8 * d * E,
                "flops": 18 * A * d * F + 4 * T * d * E}
    if kind == "route":
        return {"bytes": act + 4 * d * E + routing, "flops": 2 * T * d * E}
    if kind == "route_bwd":
        return {"bytes": act + 4 * d * E + 2 * routing, "flops": 2 * A * d}
    if kind == "dispatch":
        return {"bytes": act + 2 * A * d + routing, "flops": 0}
    if kind == "combine":
        return {"bytes": act + 2 * A * d + routing, "flops": 2 * A * d}
    if kind == "ffn_fwd":
        return {"bytes": weights + 2 * A * (2 * d + 3 * F), "flops": 6 * A * d * F}
    return {"bytes": weights + 2 * 3 * E * d * F + 2 * A * (3 * d + 5 * F) + 3 * 4 * A + 4 * d * E,
            "flops": 12 * A * d * F}


def tolerance(case):
    kind = case["kind"]
    if kind == "dispatch":
        return "exact"
    # about four times the distance from exact() that was measured: gates 1e-7 to 9.5e-6 and
    # dw_router 5e-6 (fp32 sums), 1.7e-3 (one bf16 rounding), 2.9e-3 to 3.9e-3 (a layer or
    # the FFN, two or three bf16 roundings in a row). A few indices may swap at near ties.
    if kind in ("route", "route_bwd"):
        return {"rel": 4e-5, "max": 2e-3, "differ": 1e-3}
    if kind == "combine":
        return {"rel": 7e-3}
    return {"rel": 1.4e-2, "max": 0.6, "differ": 1e-3}


# ---------------------------------------------------------------- the same in 64 bits

_MOST_FLOPS = 4e12   # what fp64 does in a few seconds
_MOST_BYTES = 24e9


def _silu64(a, b):
    s = torch.sigmoid(a)
    return a * s * b, b * (s * (1 + a * (1 - s))), a * s  # H, dH/dA, dH/dB


def _ranges(off, count):
    """(expert, first row, end of its rows) of every group with rows."""
    return [(e, o, o + n) for e, (o, n) in enumerate(zip(off.tolist()[:-1], count.tolist())) if n]


def _top(c, s):
    z = s["x"].double() @ s["w_router"].double() + s["bias"].double()
    if s["mask"] is not None:
        z[:, s["mask"] == 0] = -math.inf
    v, idx = torch.topk(z, c["k"], dim=1)
    return idx, torch.softmax(v, dim=1)


def _d_logits(gate, d_gate):
    return gate * (d_gate - (gate * d_gate).sum(1, keepdim=True))


def _router_gradient(c, x, idx, dz):
    z = torch.zeros(c["T"], c["E"], dtype=F64, device="cuda").scatter_(1, idx.long(), dz)
    return x.double().T @ z


def exact(case, seed):
    c = case
    T, d, E, k, F, R, kind = c["T"], c["d"], c["E"], c["k"], c["F"], _rows_cap(case), case["kind"]
    if work(c)["flops"] > _MOST_FLOPS or 8 * (3 * E * d * F + 2 * R * (d + 3 * F)) > _MOST_BYTES:
        return None
    s = _inputs(c, seed)
    if kind == "route":
        idx, gate = _top(c, s)
        return {"idx": idx.to(I32), "gate": gate}
    if kind == "route_bwd":
        dz = _d_logits(s["gate"].double(), s["d_gate"].double())
        return {"d_logits": dz, "dw_router": _router_gradient(c, s["x"], s["idx"], dz)}
    if kind == "dispatch":
        off, count, row = _layout(s["idx"], E)
        return {"counts": count, "off": off, "count": count, "row": row,
                "x_perm": _grouped(c, s["x"].double(), row)}
    if kind == "combine":
        y = torch.zeros(T, d, dtype=F64, device="cuda")
        for j in range(k):
            y += s["gate"][:, j:j + 1].double() * s["out_perm"][s["row"][:, j].long()].double()
        return {"y": y}

    def z64(*shape):
        return torch.zeros(*shape, dtype=F64, device="cuda")

    if kind == "ffn_fwd":
        ab, h, out = z64(R, 2 * F), z64(R, F), z64(R, d)
        for e, r0, r1 in _ranges(s["off"], s["count"]):
            ab[r0:r1] = s["x_perm"][r0:r1].double() @ s["w_gate_up"][e].double().T
            h[r0:r1] = _silu64(ab[r0:r1, :F], ab[r0:r1, F:])[0]
            out[r0:r1] = h[r0:r1] @ s["w_down"][e].double().T
        return {"ab": _block(ab), "h": h, "out": out}
    if kind == "ffn_bwd":
        d_ab, dx, dots = z64(R, 2 * F), z64(R, d), z64(R)
        dgu, ddn = z64(E, 2 * F, d), z64(E, d, F)
        groups = _ranges(s["off"], s["count"])
        for e, r0, r1 in groups:
            do, x, hh = s["d_out"][r0:r1].double(), s["x_perm"][r0:r1].double(), s["h"][r0:r1].double()
            ab = s["ab"][r0:r1].double()
            h, da, db = _silu64(ab[:, :F], ab[:, F:])
            dh = do @ s["w_down"][e].double()
            g = torch.cat([dh * da, dh * db], 1)
            d_ab[r0:r1], dots[r0:r1] = g, (dh * h).sum(1)
            dx[r0:r1] = g @ s["w_gate_up"][e].double()
            dgu[e], ddn[e] = g.T @ x, do.T @ hh
        gate = s["gate"].double()
        d_gate = dots[s["row"].long()] / gate
        dz = z64(R)
        dz[s["row"].reshape(-1).long()] = _d_logits(gate, d_gate).reshape(-1)
        for e, r0, r1 in groups:
            dx[r0:r1] += dz[r0:r1, None] * s["w_router"][:, e].double()
        return {"d_gate": d_gate, "d_ab": d_ab, "dx_perm": dx, "dw_gate_up": dgu, "dw_down": ddn}
    # a whole layer
    idx, gate = _top(c, s)
    x = s["x"].double()
    step = kind == "layer_step"
    y, dx, d_gate = z64(T, d), z64(T, d), z64(T, k)
    dgu, ddn = (z64(E, 2 * F, d), z64(E, d, F)) if step else (None, None)
    for e in range(E):
        t, j = (idx == e).nonzero(as_tuple=True)
        if t.numel() == 0:
            continue
        w1, w2, g = s["w_gate_up"][e].double(), s["w_down"][e].double(), gate[t, j][:, None]
        ab = x[t] @ w1.T
        h, da, db = _silu64(ab[:, :F], ab[:, F:])
        o = h @ w2.T
        y.index_add_(0, t, g * o)
        if step:
            dy = s["dy"][t].double()
            d_gate[t, j] = (dy * o).sum(1)
            dh = (g * dy) @ w2
            gg = torch.cat([dh * da, dh * db], 1)
            dx.index_add_(0, t, gg @ w1)
            dgu[e], ddn[e] = gg.T @ x[t], (g * dy).T @ h
    out = {"y": y, "idx": idx.to(I32), "gate": gate}
    if step:
        dz = _d_logits(gate, d_gate)
        for j in range(k):
            dx += dz[:, j:j + 1] * s["w_router"].double().T[idx[:, j]]
        out.update(dx=dx, dw_gate_up=dgu, dw_down=ddn, dw_router=_router_gradient(c, s["x"], idx, dz))
    return out
