"""The measured workloads of the library: what its users have it do, each
through a public entry point of ``paper_2211_14438_gb300.bern``.

``listed()`` names them, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` makes what a program holds before the call (weights,
boxes, result buffers; the context is one per process, as programs keep it),
``run(state)`` is one pass, ``work(case)`` the bytes and operations of the
method itself and ``exact(case, seed)`` the same results in float64.

The network shapes, orders, caps and box sides are those of
``workloads.py``, ``bench.py`` and the tests.
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_2211_14438_gb300 import bern
from paper_2211_14438_gb300 import workloads as wl

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one query box through the small two-input network: a caller that asks
        # box by box; launches and their gaps are all there is
        {"name": "single_2in", "kind": "propagate", "widths": "2-20-20-1", "boxes": 1,
         "orders": "2", "cap": 16, "lin": 0, "dist": "gauss", "cells": 0, "side_lo": 2.0,
         "side_hi": 2.0},
        # the benchmark: 4/5 grid cells, 1/5 random boxes, three inputs
        {"name": "batch_3in", "kind": "propagate", "widths": "3-64-64-64-64-1", "boxes": 5120,
         "orders": "2", "cap": 16, "lin": 0, "dist": "gauss", "cells": 16, "side_lo": 0.01,
         "side_hi": 0.5},
        # the same network from and to host buffers, the call of a program without
        # device tensors (weights and boxes in, bounds and polynomials out), on
        # boxes wide enough that every layer has unstable neurons in each: all
        # polynomials have the full term count and all of the result is written
        {"name": "batch_3in_host", "kind": "host", "widths": "3-64-64-64-64-1", "boxes": 5120,
         "orders": "2", "cap": 16, "lin": 0, "dist": "gauss", "cells": 0, "side_lo": 0.25,
         "side_hi": 0.5},
        # six inputs, wide layers, two outputs
        {"name": "batch_6in", "kind": "propagate", "widths": "6-100-100-100-2", "boxes": 2048,
         "orders": "2", "cap": 16, "lin": 0, "dist": "gauss", "cells": 0, "side_lo": 0.05,
         "side_hi": 0.5},
        # a round of children in branch and bound on the deep six-input network:
        # few boxes, polynomials of up to 74,613 terms
        {"name": "bnb_6in", "kind": "propagate", "widths": "6-64-64-64-64-1", "boxes": 48,
         "orders": "2", "cap": 16, "lin": 0, "dist": "gauss", "cells": 0, "side_lo": 0.1,
         "side_hi": 0.7},
        # orders proposed by the degree MLP, a Bernstein order per box
        {"name": "learned_3in", "kind": "learned", "widths": "3-64-64-64-64-1", "boxes": 5120,
         "orders": "4,2,2,2", "cap": 16, "lin": 0, "dist": "gauss", "cells": 16,
         "side_lo": 0.01, "side_hi": 0.5},
        # the deepest ablation network with every layer linearised
        {"name": "lin_2in", "kind": "propagate", "widths": "2-20-20-20-20-20-1", "boxes": 4096,
         "orders": "2", "cap": 64, "lin": 1, "dist": "paper", "cells": 0, "side_lo": 0.05,
         "side_hi": 0.5},
        # the ablation over the ReLU order: Horner compositions
        {"name": "orders_2in", "kind": "propagate", "widths": "2-20-20-1", "boxes": 4096,
         "orders": "4", "cap": 64, "lin": 0, "dist": "paper", "cells": 0, "side_lo": 0.05,
         "side_hi": 0.5},
        # one layer step of a caller's own pipeline: affine on ragged polynomials
        {"name": "affine_step", "kind": "affine", "n": 3, "deg": 8, "h_in": 64, "h_out": 64,
         "boxes": 2048},
        # its range enclosure at the layer's Bernstein order
        {"name": "enclose_step", "kind": "enclose", "n": 3, "deg": 8, "order": 8, "h": 64,
         "boxes": 2048},
        # and its composition with the ReLU polynomials into a new block
        {"name": "compose_step", "kind": "compose", "n": 3, "deg": 8, "h": 64, "boxes": 2048},
        # one training step of the degree MLP: backward (forward inside) and Adam,
        # the samples of 800 training boxes
        {"name": "train_step", "kind": "train", "samples": 204800, "features": 8, "classes": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    kind = rng.choice(["propagate"] * 5 + ["host", "learned", "affine", "enclose", "compose",
                                           "train"])
    if kind == "train":
        return {"kind": kind, "samples": _log_int(rng, 500, 204800),
                "features": rng.choice([8, 8, 13]), "classes": rng.choice([4, 4, 6])}
    if kind in ("affine", "enclose", "compose"):
        n = rng.choice([2, 3, 3, 4, 6])
        deg = rng.randint(1, {2: 8, 3: 8, 4: 6, 6: 4}[n])
        boxes, h = _log_int(rng, 16, 4096), rng.randint(9, 100)
        if kind == "affine":
            return {"kind": kind, "n": n, "deg": deg, "h_in": h,
                    "h_out": rng.choice([1, 2, rng.randint(9, 100)]), "boxes": boxes}
        c = {"kind": kind, "n": n, "deg": deg, "h": h, "boxes": boxes}
        return dict(c, order=deg) if kind == "enclose" else c
    lin = 0
    dist = rng.choice(["gauss", "gauss", "paper"])
    n = rng.randint(2, 6)
    layers = rng.randint(1, 4)
    hidden = [rng.randint(10, 100) if dist == "gauss" else 20] * layers
    if rng.random() < 0.4:
        hidden = [max(9, h - rng.randint(0, 9)) for h in hidden]
    outs = rng.choice([1, 1, 2])
    cap = 16 if dist == "gauss" else 64
    if kind == "learned":
        n, dist, cap = 3, "gauss", 16
        orders = ",".join(["4"] + ["2"] * (layers - 1))
    elif rng.random() < 0.7:
        orders = "2"
    else:
        orders = ",".join(str(rng.choice([1, 2, 3, 4, 5] if i == 0 else [1, 2]))
                          for i in range(layers))
    if dist == "paper" and kind == "propagate" and rng.random() < 0.4:
        n, lin, orders = min(n, 3), rng.choice([1, 2]), "2"
    if kind == "host":
        return {"kind": kind, "widths": "-".join(map(str, [n] + hidden + [outs])),
                "boxes": _log_int(rng, 2, 5120), "orders": orders, "cap": cap, "lin": 0,
                "dist": dist, "cells": 0, "side_lo": 0.25, "side_hi": 0.5}
    return {"kind": kind, "widths": "-".join(map(str, [n] + hidden + [outs])),
            "boxes": 1 if rng.random() < 0.15 else _log_int(rng, 2, 5120), "orders": orders,
            "cap": cap, "lin": lin, "dist": dist, "cells": 16 if n == 3 and rng.random() < 0.5
            else 0, "side_lo": 0.05, "side_hi": 0.5}


def _most():
    return max(work(c)["flops"] for c in listed())


def draw(rng):
    most = {"propagate": 1.0, "host": 0.2, "learned": 0.1}
    limit = _most()
    while True:
        c = _draw_once(rng)
        if "widths" in c:
            w, d = _shape(c)
            if math.prod(d) > c["cap"] and c["kind"] != "learned":
                continue   # no truncation: the orders a plan of this cap is used with
            # the whole block of a batch stays within what one call chunks well
            if c["boxes"] * max(w) * _mono(w[0], _degrees(c)[0][-1]) > 2e9:
                continue
        elif c["kind"] != "train" and c["boxes"] * max(c.get("h", 0), c.get("h_in", 0)) * _mono(
                c["n"], c["deg"] * (2 if c["kind"] == "compose" else 1)) > 2e8:
            continue
        f = work(c)
        if f["flops"] <= limit * most.get(c["kind"], 0.5) and f["bytes"] <= 2e9:
            return c


# ------------------------------------------------------------------ shapes
def _mono(n, D):
    return math.comb(n + D, n)


def _shape(case):
    widths = [int(x) for x in case["widths"].split("-")]
    d = [int(x) for x in case["orders"].split(",")]
    return widths, (d * (len(widths) - 2) if len(d) == 1 else d)


def _degrees(case):
    """Per layer the total degree of its pre-activation polynomials and the
    Bernstein order of its enclosure."""
    widths, d = _shape(case)
    D, order = [1], [1]
    for i, x in enumerate(d):
        D.append(min(D[-1] * x, case["cap"]))
        order.append(min(order[-1] * x, case["cap"]))
        if case["lin"] and (i + 1) % case["lin"] == 0:
            D[-1], order[-1] = min(widths[0], D[-1]), min(widths[0], order[-1])
    return D, order


def _grid_order(n, l, budget=1 << 20):
    while (l + 1) ** n > budget:
        l -= 1
    return min(l, 24)


# ------------------------------------------------------------------ states
@functools.lru_cache(maxsize=1)
def _context():
    return bern.Context(0, stream=torch.cuda.current_stream())


def _inputs(case, seed):
    widths, _ = _shape(case)
    rng = np.random.default_rng(seed)
    net = wl.make_net(widths, seed=seed, dist=case["dist"], rng=rng)
    n, count = widths[0], case["boxes"]
    if count == 1:
        return net, wl.box_array([-1.0] * n, [1.0] * n)[None]
    boxes = wl.random_boxes(rng, count, n, case["side_lo"], case["side_hi"])
    if case["cells"]:
        k = (4 * count) // 5
        edges = np.linspace(-1.0, 1.0, case["cells"] + 1)
        at = rng.integers(0, case["cells"], (k, n))
        boxes[:k] = wl.box_array(edges[at], edges[at + 1])
    return net, boxes


def _degree_mlp(seed):
    """An untrained degree MLP.  It weighs the features that are whole numbers
    in nature (layer, term count, stability flags), so that its proposals do
    not hang on the last bit of a bound, and leans to the low orders, as the
    trained ones do."""
    rng = np.random.default_rng(seed + 77)
    F, C, H = bern.BERN_DEGREE_FEATURES, bern.BERN_DEGREE_CLASSES, bern.BERN_MLP_HIDDEN
    W1 = rng.normal(0, np.sqrt(2.0 / F), (H, F))
    W1[:, [0, 1, 2, 7]] = 0.0
    W2 = rng.normal(0, np.sqrt(1.0 / H), (C, H))
    b2 = np.array([0.6, 0.3, -0.3, -0.6])
    theta = np.concatenate([W1.ravel(), rng.normal(0, 0.1, H), W2.ravel(), b2])
    return bern.Mlp(torch, F, C, theta)


def _ragged(case, seed, h):
    """A layer block [boxes, M, h] of both bounds in power-basis coefficients
    that fall with the degree, as layers of narrow boxes have them, and the
    term count of every neuron: the degree differs from box to box."""
    n, deg, B = case["n"], case["deg"], case["boxes"]
    M = _mono(n, deg)
    g = torch.Generator(device=DEV).manual_seed(seed)
    fall = torch.from_numpy(0.5 ** _graded(n, deg).sum(1)).to(DEV, torch.float32)
    c = torch.randn(B, M, h, device=DEV, generator=g) * fall[None, :, None]
    r = torch.randn(B, M, h, device=DEV, generator=g) * fall[None, :, None] * 0.01
    r[:, 0] = r[:, 0].abs() + 0.05
    box_deg = torch.randint(0, 4, (B,), device=DEV, generator=g)
    degs = torch.tensor([deg, deg, max(1, deg // 2), max(1, deg // 4)], device=DEV)[box_deg]
    counts = torch.tensor([_mono(n, k) for k in range(deg + 1)], device=DEV)
    nt = counts[degs][:, None].expand(B, h).clone()
    live = torch.arange(M, device=DEV)[None, :, None] < nt[:, None, :]
    return c, r, live, nt.to(torch.int32), g


def _zeros_like_results(case, host):
    widths, _ = _shape(case)
    B, o = case["boxes"], widths[-1]
    ct = _mono(widths[0], _degrees(case)[0][-1])
    if host:
        def z(shape, t):
            return torch.zeros(shape, dtype=t, pin_memory=True).numpy()
    else:
        def z(shape, t):
            return torch.zeros(shape, dtype=t, device=DEV)
    return ct, {"lo": z((B, o), torch.float32), "hi": z((B, o), torch.float32),
                "n_terms": z((B, o, 2), torch.int32), "coef": z((B, o, 2, ct), torch.float32)}


def _prepare_net(case, seed):
    widths, d = _shape(case)
    net, boxes = _inputs(case, seed)
    host = case["kind"] == "host"
    ct, out = _zeros_like_results(case, host)
    if host:
        pin = torch.from_numpy(boxes).pin_memory()
        W, b, bx = net.W, net.b, pin.numpy()
    else:
        W = [torch.from_numpy(x).to(DEV) for x in net.W]
        b = [torch.from_numpy(x).to(DEV) for x in net.b]
        bx = torch.from_numpy(boxes).to(DEV)
    degree = d if len(set(d)) > 1 else d[0] if d else 2
    if case["kind"] == "learned":
        degree = bern.Learned(_degree_mlp(seed), max_per_layer=d)
    return {"widths": widths, "W": W, "b": b, "boxes": bx, "degree": degree, "out": out,
            "cap_terms": ct}


def _prepare_affine(case, seed):
    B, h, ho = case["boxes"], case["h_in"], case["h_out"]
    c, r, live, nt, g = _ragged(case, seed, h)
    # dead neurons hold no term, the rest a graded prefix of their own
    pick = torch.rand(B, h, device=DEV, generator=g)
    nt = torch.where(pick < 0.25, torch.zeros_like(nt), nt)
    nt = torch.where((pick > 0.85), nt.clamp(max=case["n"] + 1), nt)
    M = c.shape[1]
    W = torch.randn(ho, h, device=DEV, generator=g) / math.sqrt(h)
    b = torch.rand(ho, device=DEV, generator=g) * 0.2 - 0.1
    return {"W": W, "b": b, "up": c + r, "lo": c - r, "nt": nt,
            "out_up": torch.zeros(B, M, ho, device=DEV),
            "out_lo": torch.zeros(B, M, ho, device=DEV),
            "out_nt": torch.zeros(B, ho, dtype=torch.int32, device=DEV)}


def _prepare_enclose(case, seed):
    c, r, live, nt, _ = _ragged(case, seed, case["h"])
    z = torch.zeros(case["boxes"], case["h"], device=DEV)
    return {"up": (c + r) * live, "lo": (c - r) * live, "nt": nt, "res_lo": z,
            "res_hi": z.clone()}


def _prepare_compose(case, seed):
    h, B = case["h"], case["boxes"]
    c, r, live, nt, _ = _ragged(case, seed, h)
    up, lo = (c + r) * live, (c - r) * live
    # a third of the neurons each dead, active and unstable, by the constant
    third = torch.arange(h, device=DEV) % 3
    span = c.abs().mul(live)[:, 1:].sum(1)
    move = torch.where(third == 0, -2.0 * span - 1.0, torch.where(third == 1, 2.0 * span + 1.0,
                                                                  0.0 * span))
    up[:, 0] += move
    lo[:, 0] += move
    L = (lo[:, 0].double() + lo[:, 1:].clamp(max=0).double().sum(1)).float() - 1e-3
    H = (up[:, 0].double() + up[:, 1:].clamp(min=0).double().sum(1)).float() + 1e-3
    kind = torch.where(H <= 0, 0, torch.where(L >= 0, 1, 2)).to(torch.int8)
    # order 2 in closed form: (lo + hi) s - lo s^2, or hi s^2
    pos = L + H > 0
    coef = torch.zeros(B, h, bern.COEF_STRIDE, device=DEV)
    coef[..., 1] = torch.where(pos, L + H, torch.zeros_like(L))
    coef[..., 2] = torch.where(pos, -L, H)
    w2 = (H - L) ** 2
    eps = torch.where(pos, -L * H * H, H * L * L) / w2 * (1 + 1e-6) + 1e-6
    M2 = _mono(case["n"], 2 * case["deg"])
    return {"up": up, "lo": lo, "nt": nt, "L": L, "H": H, "kind": kind, "coef": coef, "eps": eps,
            "post_up": torch.zeros(B, M2, h, device=DEV),
            "post_lo": torch.zeros(B, M2, h, device=DEV),
            "post_nt": torch.zeros(B, h, dtype=torch.int32, device=DEV)}


def _prepare_train(case, seed):
    F, C, H, N = case["features"], case["classes"], bern.BERN_MLP_HIDDEN, case["samples"]
    rng = np.random.default_rng(seed)
    P = int(bern.load().bern_mlp_num_params(F, C))
    theta = np.zeros(P, np.float32)
    theta[:H * F] = rng.normal(0, np.sqrt(2.0 / F), H * F)
    o = H * F + H
    theta[o:o + C * H] = rng.normal(0, np.sqrt(1.0 / H), C * H)
    mlp = bern.Mlp(torch, F, C, theta)
    g = torch.Generator(device=DEV).manual_seed(seed)
    X = torch.rand(N, F, device=DEV, generator=g) * 2.0 - 1.0
    y = torch.multinomial(torch.tensor([0.6, 0.3, 0.06, 0.04, 0.02, 0.02][:C], device=DEV), N,
                          True, generator=g).to(torch.int32)
    return {"mlp": mlp, "X": X, "y": y, "grad": torch.zeros(P, device=DEV),
            "loss": torch.zeros(1, device=DEV)}


_PREPARE = {"affine": _prepare_affine, "enclose": _prepare_enclose, "compose": _prepare_compose,
            "train": _prepare_train}


def prepare(case, seed):
    s = _PREPARE.get(case["kind"], _prepare_net)(case, seed)
    return dict(s, case=case, ctx=_context())


# ------------------------------------------------------------------ one pass
def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "host":
        return ctx.propagate_host(s["widths"], s["W"], s["b"], s["boxes"], degree=s["degree"],
                                  cap=case["cap"], cap_terms=s["cap_terms"], out=s["out"],
                                  lin=case["lin"])
    if "widths" in s:
        return ctx.propagate(s["widths"], s["W"], s["b"], s["boxes"], degree=s["degree"],
                             cap=case["cap"], cap_terms=s["cap_terms"], out=s["out"],
                             sync=False, lin=case["lin"])
    if kind == "affine":
        M = s["up"].shape[1]
        ctx.affine(case["boxes"], case["h_out"], case["h_in"], s["W"], s["b"], s["up"], s["lo"],
                   M, s["nt"], s["out_up"], s["out_lo"], M, s["out_nt"])
        return {"up": s["out_up"], "lo": s["out_lo"], "n_terms": s["out_nt"]}
    if kind == "enclose":
        ctx.enclose(case["n"], case["boxes"], case["h"], case["order"], 0, s["up"], s["lo"],
                    s["up"].shape[1], s["nt"], s["res_lo"], s["res_hi"])
        return {"lo": s["res_lo"], "hi": s["res_hi"]}
    if kind == "compose":
        ctx.compose(case["n"], case["boxes"], case["h"], 2 * case["deg"], 0.0, s["kind"],
                    s["coef"], s["eps"], None, 2, s["L"], s["H"], s["up"], s["lo"],
                    s["up"].shape[1], s["nt"], s["post_up"], s["post_lo"], s["post_up"].shape[1],
                    s["post_nt"])
        return {"up": s["post_up"], "lo": s["post_lo"], "n_terms": s["post_nt"]}
    m = s["mlp"]
    ctx.mlp_backward(m, s["X"], s["y"], None, s["grad"], s["loss"])
    ctx.mlp_adam(m, s["grad"], 3e-3)
    return {"grad": s["grad"], "loss": s["loss"], "param": m.param, "m": m.m, "v": m.v,
            "W1": m.W1.view(torch.bfloat16), "W2": m.W2.view(torch.bfloat16)}


# ------------------------------------------------------------------ its work
def _enclose_flops(n, l):
    lines = sum(math.comb(l + k, k) * (l + 1) ** (n - 1 - k) for k in range(n))
    return 2 * lines * (l * (l + 1) // 2)


def work(case):
    """Inputs read once, outputs written once; the method's multiply-adds, two
    operations each.  Of a network's hidden neurons half are taken to be
    unstable (enclosed and composed); of a ragged block half the terms.  A
    learned plan counts as one of order 2: its proposals lean below its caps."""
    kind = case["kind"]
    if kind == "learned":
        case = dict(case, orders="2")
    if kind == "train":
        N, F, C, H = case["samples"], case["features"], case["classes"], bern.BERN_MLP_HIDDEN
        return {"bytes": 4 * N * (F + 1), "flops": 2 * N * H * (2 * F + 3 * C)}
    if "widths" not in case:
        n, deg, B = case["n"], case["deg"], case["boxes"]
        M = _mono(n, deg)
        if kind == "affine":
            return {"bytes": 4 * B * M * (case["h_in"] + case["h_out"]),
                    "flops": 2 * B * M * case["h_in"] * case["h_out"]}
        h = case["h"]
        if kind == "enclose":
            return {"bytes": 4 * B * h * M, "flops": B * h * _enclose_flops(n, case["order"])}
        return {"bytes": 4 * B * h * (2 * M + _mono(n, 2 * deg)) // 3,
                "flops": B * h * M * (M + 1) // 3}
    widths, d = _shape(case)
    n, B = widths[0], case["boxes"]
    D, order = _degrees(case)
    flops = 0
    for i in range(len(widths) - 1):
        M = _mono(n, D[i])
        flops += 4 * widths[i] * widths[i + 1] * M
        share = 0.5 if i < len(d) else 1.0
        flops += 2 * share * widths[i + 1] * _enclose_flops(n, _grid_order(n, order[i]))
        if i < len(d):
            pairs = (M * (M + 1) / 2 if d[i] == 2 else
                     sum(_mono(n, D[i] * k) * M for k in range(1, d[i])))
            flops += 4 * share * widths[i + 1] * pairs
            if case["lin"] and (i + 1) % case["lin"] == 0:
                flops += 2 * widths[i + 1] * _enclose_flops(n, D[i] * d[i])
    weights = sum(a * (b + 1) for a, b in zip(widths[1:], widths))
    bytes_ = 4 * (weights + B * (2 * n + widths[-1] * (4 + 2 * _mono(n, D[-1]))))
    return {"bytes": bytes_, "flops": B * flops}


# ------------------------------------------------------------------ float64
@functools.lru_cache(maxsize=64)
def _graded(n, D):
    """Exponents of total degree <= D: by degree, then descending."""
    def of(n, d):
        if n == 1:
            return [(d,)]
        return [(a,) + t for a in range(d, -1, -1) for t in of(n - 1, d - a)]
    return np.array([e for d in range(D + 1) for e in of(n, d)], np.int64)


@functools.lru_cache(maxsize=64)
def _product_index(n, Dq, Ds):
    """[M(n, Dq), M(n, Ds)]: the rank of the product of two monomials."""
    w = (Dq + Ds + 1) ** np.arange(n, dtype=np.int64)
    keys = _graded(n, Dq + Ds) @ w
    by = np.argsort(keys)
    both = (_graded(n, Dq) @ w)[:, None] + (_graded(n, Ds) @ w)[None]
    return torch.from_numpy(by[np.searchsorted(keys[by], both)]).to(DEV)


def _mul(n, q, Dq, s, Ds):
    """Products of polynomials, items x coefficients."""
    ix = _product_index(n, Dq, Ds)
    out = torch.zeros(q.shape[0], _mono(n, Dq + Ds), dtype=q.dtype, device=DEV)
    for J in range(s.shape[1]):
        out.index_add_(1, ix[:, J].contiguous(), q * s[:, J:J + 1])
    return out


def _range(n, P, D, l, want):
    """max (want 1) or min (want -1) of the Bernstein coefficients of order l
    of the polynomials P [items, M(n, D)], with the terms above the order at
    their own intervals."""
    e = _graded(n, D)
    low = e.sum(1) <= l
    scale = np.array([math.prod(math.comb(l, int(j)) for j in t) for t in e[low]], np.float64)
    cell = torch.from_numpy((e[low] * ((l + 1) ** np.arange(n - 1, -1, -1))).sum(1)).to(DEV)
    T = torch.tensor([[float(math.comb(i, j)) for j in range(l + 1)] for i in range(l + 1)],
                     dtype=torch.float64, device=DEV)
    a = P[:, torch.from_numpy(low).to(DEV)] / torch.from_numpy(scale).to(DEV)
    rest = P[:, torch.from_numpy(~low).to(DEV)] * want
    got = rest.clamp(min=0).sum(1) * want
    step = max(1, (1 << 27) // (l + 1) ** n)
    for i in range(0, P.shape[0], step):
        part = a[i:i + step]
        grid = torch.zeros(part.shape[0], (l + 1) ** n, dtype=torch.float64, device=DEV)
        grid[:, cell] = part
        grid = grid.reshape([-1] + [l + 1] * n)
        for k in range(n):
            grid = torch.tensordot(grid, T, dims=([1], [1]))   # the axis moves to the end
        grid = grid.reshape(part.shape[0], -1)
        got[i:i + step] += grid.amax(1) if want > 0 else grid.amin(1)
    return got


def _relu_power(L, H, d):
    """The order-d Bernstein polynomial of ReLU on [L, H] in powers of s, and
    its value at the s of 0."""
    w = H - L
    b = [(L + w * (k / d)).clamp(min=0) for k in range(d + 1)]
    a = [sum(b[k] * (math.comb(d, k) * math.comb(d - k, j - k) * (-1) ** (j - k))
             for k in range(j + 1)) for j in range(d + 1)]
    s0 = -L / w
    return a, sum(b[k] * math.comb(d, k) * s0 ** k * (1 - s0) ** (d - k) for k in range(d + 1))


def _compose(n, P, D, L, H, a):
    """B(s) with s = (P - L) / (H - L), items x coefficients."""
    s = P.clone()
    s[:, 0] -= L
    s /= (H - L)[:, None]
    q, Dq = a[-1][:, None].clone(), 0
    for aj in a[-2::-1]:
        q, Dq = _mul(n, q, Dq, s, D), Dq + D
        q[:, 0] += aj
    return q


def _multilinear(n, D):
    """The least-squares multilinear fit of every monomial, as a matrix onto
    the monomials of degree <= min(n, D)."""
    e, f = _graded(n, D), _graded(n, min(n, D))
    beta = 6.0 * e / ((e + 1) * (e + 2))
    alpha = 1.0 / (e + 1) - beta / 2
    A = np.zeros((len(e), len(f)))
    for c, t in enumerate(f):
        if t.max(initial=0) <= 1:
            A[:, c] = np.prod(np.where(t[None] == 1, beta, alpha), axis=1)
    return torch.from_numpy(A).to(DEV)


def _pad(P, M):
    return torch.nn.functional.pad(P, (0, M - P.shape[-1]))


def _exact_boxes(case, W, b, boxes):
    """Bounds and polynomials of some boxes."""
    widths, d = _shape(case)
    n, B = widths[0], boxes.shape[0]
    D, order = _degrees(case)
    up = torch.zeros(B, n, n + 1, dtype=torch.float64, device=DEV)
    up[:, :, 0] = boxes[..., 0]
    up[:, torch.arange(n), torch.arange(1, n + 1)] = boxes[..., 1] - boxes[..., 0]
    lo = up.clone()
    for i in range(len(widths) - 1):
        pos, neg = W[i].clamp(min=0), W[i].clamp(max=0)
        up, lo = pos @ up + neg @ lo, pos @ lo + neg @ up
        up[:, :, 0] += b[i]
        lo[:, :, 0] += b[i]
        h, M = widths[i + 1], _mono(n, D[i])
        l = _grid_order(n, order[i])
        fu, fl = up.reshape(B * h, M), lo.reshape(B * h, M)
        H, L = _range(n, fu, D[i], l, 1), _range(n, fl, D[i], l, -1)
        if i == len(d):
            return L.reshape(B, h), H.reshape(B, h), torch.stack([up, lo], 2)
        dead, un = H <= 0, (L < 0) & (H > 0)
        Dp = D[i] * d[i]
        Mp = _mono(n, Dp)
        pu, pl = _pad(fu, Mp).clone(), _pad(fl, Mp).clone()
        pu[dead], pl[dead] = 0.0, 0.0
        at = torch.nonzero(un)[:, 0]
        step = max(1, (1 << 28) // Mp)
        for k in range(0, at.numel(), step):
            x = at[k:k + step]
            a, eps = _relu_power(L[x], H[x], d[i])
            pu[x] = _compose(n, fu[x], D[i], L[x], H[x], a)
            q = _compose(n, fl[x], D[i], L[x], H[x], a)
            q[:, 0] -= eps
            pl[x] = q
        if case["lin"] and (i + 1) % case["lin"] == 0:
            A = _multilinear(n, Dp)
            l2 = _grid_order(n, min(order[i] * d[i], case["cap"]))
            au, al = pu @ A, pl @ A
            Ml = A.shape[1]
            au[:, 0] += torch.where(dead, 0.0, _range(n, pu - _pad(au, Mp), Dp, l2, 1))
            al[:, 0] += torch.where(dead, 0.0, _range(n, pl - _pad(al, Mp), Dp, l2, -1))
            pu, pl, Mp = au, al, Ml
        up, lo = pu.reshape(B, h, Mp), pl.reshape(B, h, Mp)


def _exact_net(case, seed):
    if case["kind"] == "learned":
        return None   # the orders are the outcome of a bf16 network
    widths, d = _shape(case)
    net, boxes = _inputs(case, seed)
    W = [torch.from_numpy(x).to(DEV, torch.float64) for x in net.W]
    b = [torch.from_numpy(x).to(DEV, torch.float64) for x in net.b]
    bx = torch.from_numpy(boxes).to(DEV, torch.float64)
    D = _degrees(case)[0]
    big = max(w * _mono(widths[0], x) for w, x in zip(widths[1:], D[1:] + D[-1:]))
    step = max(1, (1 << 28) // big)
    parts = [_exact_boxes(case, W, b, bx[i:i + step]) for i in range(0, len(boxes), step)]
    lo, hi, coef = (torch.cat(p) for p in zip(*parts))
    return {"lo": lo, "hi": hi, "n_terms": None, "coef": coef}


def _exact_affine(s):
    live = torch.arange(s["up"].shape[1], device=DEV)[None, :, None] < s["nt"][:, None, :]
    u, l = s["up"].double() * live, s["lo"].double() * live
    pos, neg = s["W"].double().clamp(min=0).T, s["W"].double().clamp(max=0).T
    up, lo = u @ pos + l @ neg, l @ pos + u @ neg
    up[:, 0] += s["b"]
    lo[:, 0] += s["b"]
    kept = torch.arange(u.shape[1], device=DEV)[None, :, None] < s["nt"].amax(1).clamp(
        min=1)[:, None, None]
    return {"up": up * kept, "lo": lo * kept, "n_terms": None}


def _rows(P):
    return P.double().transpose(1, 2).reshape(-1, P.shape[1])


def _exact_enclose(s):
    c = s["case"]
    shape = (c["boxes"], c["h"])
    return {"lo": _range(c["n"], _rows(s["lo"]), c["deg"], c["order"], -1).reshape(shape),
            "hi": _range(c["n"], _rows(s["up"]), c["deg"], c["order"], 1).reshape(shape)}


def _exact_compose(s):
    c = s["case"]
    n, D, h, B = c["n"], c["deg"], c["h"], c["boxes"]
    M2 = _mono(n, 2 * D)
    L, H = s["L"].double().reshape(-1), s["H"].double().reshape(-1)
    kind, coef = s["kind"].reshape(-1), s["coef"].double().reshape(B * h, -1)
    out = {"n_terms": None}
    for name, shift in (("up", 0.0), ("lo", 1.0)):
        P = _rows(s[name])
        got = torch.zeros(B * h, M2, dtype=torch.float64, device=DEV)
        same = kind == 1
        got[same] = _pad(P[same], M2)
        at = torch.nonzero(kind == 2)[:, 0]
        for x in at.split(max(1, (1 << 28) // M2)):
            q = _compose(n, P[x], D, L[x], H[x], [coef[x, j] for j in range(3)])
            q[:, 0] -= shift * s["eps"].double().reshape(-1)[x]
            got[x] = q
        out[name] = got.reshape(B, h, M2).transpose(1, 2)
    return out


def _exact_train(s):
    m, c = s["mlp"], s["case"]
    F, C, H, N = c["features"], c["classes"], bern.BERN_MLP_HIDDEN, c["samples"]
    W1 = m.W1.view(torch.bfloat16).double().reshape(H, F)
    W2 = m.W2.view(torch.bfloat16).double().reshape(C, H)
    x = s["X"].to(torch.bfloat16).double()
    pre = x @ W1.T + m.b1.double()
    a = pre.clamp(min=0).float().to(torch.bfloat16).double()
    z = a @ W2.T + m.b2.double()
    y = s["y"].long()
    loss = -torch.log_softmax(z, 1).gather(1, y[:, None]).mean().reshape(1)
    dz = torch.softmax(z, 1)
    dz[torch.arange(N, device=DEV), y] -= 1.0
    dh = (dz @ W2) * (pre > 0)
    grad = torch.cat([(dh.T @ x).reshape(-1), dh.sum(0), (dz.T @ a).reshape(-1), dz.sum(0)]) / N
    mm, v = 0.1 * grad, 0.001 * grad ** 2
    param = m.param.double() - 3e-3 * (mm / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    o = H * F + H
    return {"grad": grad, "loss": loss, "param": param, "m": mm, "v": v, "W1": param[:H * F],
            "W2": param[o:o + C * H]}


def exact(case, seed):
    kind = case["kind"]
    if kind not in _PREPARE:
        return _exact_net(case, seed)
    return {"affine": _exact_affine, "enclose": _exact_enclose, "compose": _exact_compose,
            "train": _exact_train}[kind](dict(_PREPARE[kind](case, seed), case=case))
