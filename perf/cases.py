"""The work a user has this library do, as timed cases.

Every case goes through the public entry points of
``paper_1410_7922_gb300.edp`` (and ``proposal``): EDP solves of stereo and
motion pairs from a cost volume or from the images, the scanline DP, the
coarse-to-fine windowed path, a batch of mixed problems, and the proposal
network's inference and training step.  ``listed()`` names the cases,
``draw()`` gives further ones of the same ranges, ``prepare()`` makes what a
program holds before the call, ``run()`` is one pass, ``work()`` what a pass
cannot do without, and ``exact()`` the same results from plain numpy / torch
in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

# Two-axis label spaces of the repository's workloads and tests, and ragged ones.
MOTION_SHAPES = [(9, 9), (17, 17), (25, 25), (33, 33), (27, 15), (20, 12), (21, 13), (31, 19)]
BATCH_SIZES = [(160, 120), (240, 180), (320, 240)]


def listed() -> list[dict]:
    return [
        # the smallest call: a thumbnail stereo pair, images to labels and energy
        dict(name="stereo_images_64x48_q16", kind="edp", W=64, H=48, Q0=16, Q1=1, Q2=1, lam=20, g=4, l1=1,
             mode="joint", iters=1, images=True, weighted=False),
        # the Cones-sized stereo pair, cost volume in hand
        dict(name="stereo_450x375_q64", kind="edp", W=450, H=375, Q0=64, Q1=1, Q2=1, lam=20, g=4, l1=1,
             mode="joint", iters=1, images=False, weighted=False),
        # the paper's second setup: 60 disparities, quadratic prior, more than one iteration
        dict(name="stereo_quadratic_450x375_q60", kind="edp", W=450, H=375, Q0=60, Q1=1, Q2=1, lam=20, g=3, l1=2,
             mode="joint", iters=2, images=False, weighted=False),
        # motion between video frames, 33 x 33 offsets, cost volume in hand
        dict(name="motion_320x240_33x33", kind="edp", W=320, H=240, Q0=33, Q1=33, Q2=1, lam=15, g=3, l1=1,
             mode="per_axis", iters=1, images=False, weighted=False),
        # the paper's third setup (Back Yard): 27 x 15 offsets, joint truncation, from the images
        dict(name="motion_images_320x265_27x15", kind="edp", W=320, H=265, Q0=27, Q1=15, Q2=1, lam=15, g=3, l1=1,
             mode="joint", iters=1, images=True, weighted=False),
        # the largest: a full VGA motion pair over 65 x 65 offsets, images to labels and energy
        dict(name="motion_images_640x480_65x65", kind="edp", W=640, H=480, Q0=65, Q1=65, Q2=1, lam=15, g=3, l1=1,
             mode="per_axis", iters=1, images=True, weighted=False),
        # motion and disparity at once with a third image
        dict(name="motion_stereo_240x180_17x17x9", kind="edp", W=240, H=180, Q0=17, Q1=17, Q2=9, lam=15, g=3, l1=1,
             mode="per_axis", iters=1, images=True, weighted=False),
        # per-row DP with back-tracking over a stereo cost volume
        dict(name="scanline_450x375_q64", kind="scanline", W=450, H=375, Q0=64, lam=20, g=4, marginals=False),
        # coarse-to-fine motion: coarse labels, then EDP on a 9 x 9 box around each
        dict(name="windowed_640x480_9x9", kind="windowed", W=640, H=480, Q0=65, win=9),
        # many small problems of mixed sizes and label spaces in one call
        dict(name="batch_12_mixed", kind="batch", n=12, max_size=2, mix=0),
        # the proposal network on one VGA frame
        dict(name="net_forward_1x480x640", kind="net", N=1, H=480, W=640, train=False),
        # one training step of the proposal network: forward, backward, Adam
        dict(name="net_train_8x240x320", kind="net", N=8, H=240, W=320, train=True),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    kind = rng.choice(["stereo", "stereo", "motion", "motion", "motion65", "volume", "scanline", "windowed", "batch",
                       "net", "net"])
    base = dict(kind="edp", Q2=1, iters=rng.choice([1, 1, 2]), weighted=False)
    if kind == "stereo":
        l1 = rng.choice([1, 1, 2])
        return dict(base, W=_log_int(rng, 48, 640), H=_log_int(rng, 36, 480), Q0=_log_int(rng, 12, 256), Q1=1,
                    lam=rng.randint(5, 30), g=rng.randint(2, 8) if l1 == 1 else rng.randint(2, 4), l1=l1,
                    mode="joint", images=rng.random() < 0.4, weighted=rng.random() < 0.2)
    if kind == "motion":
        Q0, Q1 = rng.choice(MOTION_SHAPES)
        W, H = _log_int(rng, 64, 320), _log_int(rng, 48, 265)
        return dict(base, W=W, H=H, Q0=Q0, Q1=Q1, lam=rng.randint(5, 30), g=rng.randint(2, 6), l1=1,
                    mode=rng.choice(["per_axis", "joint"]), images=rng.random() < 0.5,
                    iters=base["iters"] if W * H <= 30000 else 1)
    if kind == "motion65":
        return dict(base, W=_log_int(rng, 96, 480), H=_log_int(rng, 64, 400), Q0=65, Q1=65, iters=1,
                    lam=rng.randint(5, 30), g=rng.randint(2, 6), l1=1, mode=rng.choice(["per_axis", "joint"]),
                    images=rng.random() < 0.5)
    if kind == "volume":
        Q0, Q1, Q2 = rng.choice([(17, 17, 9), (9, 9, 9), (9, 9, 5), (11, 7, 5)])
        return dict(base, W=_log_int(rng, 48, 240), H=_log_int(rng, 36, 180), Q0=Q0, Q1=Q1, Q2=Q2, iters=1,
                    lam=rng.randint(5, 30), g=rng.randint(2, 5), l1=1, mode=rng.choice(["per_axis", "joint"]),
                    images=True)
    if kind == "scanline":
        return dict(kind="scanline", W=_log_int(rng, 64, 640), H=_log_int(rng, 48, 480), Q0=_log_int(rng, 12, 256),
                    lam=rng.randint(5, 30), g=rng.randint(2, 8), marginals=rng.random() < 0.4)
    if kind == "windowed":
        return dict(kind="windowed", W=_log_int(rng, 96, 640), H=_log_int(rng, 72, 480),
                    Q0=rng.choice([33, 65]), win=rng.choice([5, 7, 9, 11, 13, 15]))
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(4, 8), max_size=rng.randint(1, 2), mix=rng.randint(1, 1000))
    return dict(kind="net", N=rng.randint(1, 8), H=_log_int(rng, 60, 240), W=_log_int(rng, 80, 320),
                train=rng.random() < 0.5)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _texture(rng, H: int, W: int) -> np.ndarray:
    """Smoothed noise stretched to 0..255 (float32)."""
    t = rng.random((H + 8, W + 8), dtype=np.float32)
    for _ in range(2):
        t = (t[:-2] + t[1:-1] + t[2:]) / 3
        t = (t[:, :-2] + t[:, 1:-1] + t[:, 2:]) / 3
    t = t[:H, :W]
    t = t - t.min()
    return t * (255.0 / max(float(t.max()), 1e-6))


def _u8(rng, img: np.ndarray) -> np.ndarray:
    noise = rng.normal(0.0, 2.0, img.shape)
    return np.clip(np.rint(img + noise), 0, 255).astype(np.uint8)


def _shifted(rng, I0: np.ndarray, lo: tuple, hi: tuple) -> np.ndarray:
    """I1 with I1(p + v) = I0(p): a background and a few rectangles, each with
    a constant displacement v between lo and hi (x, y)."""
    H, W = I0.shape
    yy, xx = np.mgrid[0:H, 0:W]
    out = np.empty_like(I0)
    for k in range(4):
        dx, dy = int(rng.integers(lo[0], hi[0] + 1)), int(rng.integers(lo[1], hi[1] + 1))
        src = I0[np.clip(yy - dy, 0, H - 1), np.clip(xx - dx, 0, W - 1)]
        if k == 0:
            out[:] = src
            continue
        x0, y0 = int(rng.integers(0, W)), int(rng.integers(0, H))
        x1, y1 = x0 + max(1, W // 3), y0 + max(1, H // 3)
        out[y0:y1, x0:x1] = src[y0:y1, x0:x1]
    return out


def _space(Q0: int, Q1: int, Q2: int) -> dict:
    if Q2 > 1:
        return {"R": 3, "Q": (Q0, Q1, Q2), "vmin": (-(Q0 // 2), -(Q1 // 2), 0), "step": (1, 1, -1)}
    if Q1 > 1:
        return {"R": 2, "Q": (Q0, Q1, 1), "vmin": (-(Q0 // 2), -(Q1 // 2), 0), "step": (1, 1, 1)}
    return {"R": 1, "Q": (Q0, 1, 1), "vmin": (0, 0, 0), "step": (-1, 1, 1)}


def _images(seed: int, W: int, H: int, space: dict):
    """(I0, I1, I2 or None) as uint8 arrays."""
    rng = np.random.default_rng(seed)
    tex = _texture(rng, H, W)
    Q = space["Q"]
    if space["R"] == 1:
        I1 = _shifted(rng, tex, (-(Q[0] - 1), 0), (0, 0))
    else:
        r0, r1 = Q[0] // 2, Q[1] // 2
        I1 = _shifted(rng, tex, (-r0, -r1), (r0, r1))
    I2 = _u8(rng, _shifted(rng, tex, (-(Q[2] - 1), 0), (0, 0))) if space["R"] == 3 else None
    return _u8(rng, tex), _u8(rng, I1), I2


def _edp_inputs(case: dict, seed: int) -> dict:
    space = _space(case["Q0"], case.get("Q1", 1), case.get("Q2", 1))
    prior = {"lam": case["lam"], "g": case["g"], "l1": case.get("l1", 1), "mode": case.get("mode", "joint")}
    I0, I1, I2 = _images(seed, case["W"], case["H"], space)
    return {"space": space, "prior": prior, "l2": 1, "cmax": 20, "I0": I0, "I1": I1, "I2": I2,
            "cost_mode": "pair_stereo3" if I2 is not None else "pair"}


def _batch_items(case: dict, seed: int) -> list[dict]:
    """The problems of a batch: the mix (sizes and label spaces) belongs to the
    case, the images to the seed."""
    pick = np.random.default_rng(case["mix"])
    items = []
    for k in range(case["n"]):
        W, H = BATCH_SIZES[int(pick.integers(0, case["max_size"] + 1))]
        if k % 3 == 0:
            shape, lam, g, mode = (int(pick.choice([32, 48, 64, 96, 128])), 1, 1), 20, 4, "joint"
        elif k % 3 == 1:
            q = int(pick.choice([17, 25, 33]))
            shape, lam, g, mode = (q, q, 1), 15, 3, "per_axis"
        else:
            shape, lam, g, mode = (17, 17, 9) if k < 6 else (9, 9, 9), 15, 3, "per_axis"
        c = dict(W=W, H=H, Q0=shape[0], Q1=shape[1], Q2=shape[2], lam=lam, g=g, l1=1, mode=mode)
        items.append(dict(_edp_inputs(c, seed * 1000 + k), W=W, H=H))
    return items


NET_CHANNELS = (5, 32, 32, 32, 32, 32, 2)
ADAM = dict(lr=2e-3, b1=0.9, b2=0.999, eps=1e-8, step=3)


def _net_inputs(case: dict, seed: int) -> dict:
    """Parameters (He-uniform weights, small biases), features, targets and
    optimiser state on the CPU."""
    g = torch.Generator().manual_seed(seed)
    parts = []
    for ci, co in zip(NET_CHANNELS[:-1], NET_CHANNELS[1:]):
        parts.append((torch.rand(co * ci * 9, generator=g) * 2 - 1) * math.sqrt(6.0 / (ci * 9)))
        parts.append((torch.rand(co, generator=g) - 0.5) * 0.1)
    N, H, W = case["N"], case["H"], case["W"]
    P = torch.cat(parts)
    x = torch.rand((N, H, W, 5), generator=g)
    x[..., 2:4] = x[..., 2:4] * 4 - 2  # label coordinates, centred and scaled
    t = torch.randn((N, H, W, 2), generator=g) * 2
    m = torch.randn(P.shape, generator=g) * 1e-3
    v = torch.rand(P.shape, generator=g) * 1e-5
    return {"P": P, "x": x.to(torch.bfloat16), "t": t, "m": m, "v": v}


def prepare(case: dict, seed: int) -> dict:
    from paper_1410_7922_gb300 import edp

    def dev(a):
        return None if a is None else torch.as_tensor(a).cuda()

    kind = case["kind"]
    st = {"case": case}
    if kind in ("edp", "scanline"):
        w = _edp_inputs(case, seed)
        W, H = case["W"], case["H"]
        for k in ("space", "prior", "l2", "cmax", "cost_mode"):
            st[k] = w[k]
        for k in ("I0", "I1", "I2"):
            st[k] = dev(w[k])
        if not case.get("images"):
            st["C"] = edp.cost_volume(st["I0"], st["I1"], st["I2"], w["space"], w["l2"], w["cmax"], w["cost_mode"])
        if case.get("weighted"):
            st["wh"], st["wv"] = edp.edge_weights(st["I0"])
        if kind == "scanline":
            op = edp.OP_SCANLINE_MARGINALS if case["marginals"] else edp.OP_SCANLINE_DP
            st["ws"] = edp.workspace(op, W, H, w["space"], w["prior"])
        else:
            op = edp.OP_SOLVE_IMAGES if case["images"] and not case["weighted"] else edp.OP_SOLVE
            st["ws"] = edp.workspace(op, W, H, w["space"], w["prior"], case["iters"])
    elif kind == "windowed":
        from paper_1410_7922_gb300 import proposal
        w = proposal.pair_meta(case["W"], case["H"], case["Q0"] // 2)
        I0, I1, _ = _images(seed, case["W"], case["H"], w["space"])
        st.update(w=w, I0=dev(I0), I1=dev(I1))
        st["ws_c"] = edp.workspace(edp.OP_COARSE, case["W"], case["H"], w["space"], w["prior"], 1, l2=w["l2"],
                                   cmax=w["cmax"])
        st["ws_w"] = edp.workspace_windowed(case["W"], case["H"], w["space"], w["prior"], case["win"], 1)
    elif kind == "batch":
        items = []
        for it in _batch_items(case, seed):
            d = dict(it, I0=dev(it["I0"]), I1=dev(it["I1"]), I2=dev(it["I2"]), iters=1)
            d["labels"] = torch.empty((it["H"], it["W"]), dtype=torch.int32, device="cuda")
            d["energy4"] = torch.empty(4, dtype=torch.int64, device="cuda")
            items.append(d)
        st["items"] = items
        st["problems"] = edp.make_problems(items)
        st["ws"] = torch.empty(edp.batch_workspace_size(st["problems"]), dtype=torch.uint8, device="cuda")
    else:
        for k, v in _net_inputs(case, seed).items():
            st[k] = v.cuda()
        st["ws"] = edp.net_workspace(case["N"], case["H"], case["W"])
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st: dict):
    from paper_1410_7922_gb300 import edp
    case = st["case"]
    kind = case["kind"]
    if kind == "edp":
        space, prior, it = st["space"], st["prior"], case["iters"]
        if case["weighted"]:
            C = st.get("C")
            if C is None:
                C = edp.cost_volume(st["I0"], st["I1"], st["I2"], space, st["l2"], st["cmax"], st["cost_mode"])
            lab = edp.solve_weighted(C, space, prior, st["wh"], st["wv"], 2, iters=it, ws=st["ws"])
            return lab, edp.energy_weighted(C, lab, space, prior, st["wh"], st["wv"])
        if case["images"]:
            return edp.solve_images(st["I0"], st["I1"], st["I2"], space, prior, st["l2"], st["cmax"],
                                    st["cost_mode"], iters=it, ws=st["ws"])
        return (edp.solve(st["C"], space, prior, iters=it, ws=st["ws"]),)
    if kind == "scanline":
        if case["marginals"]:
            return edp.scanline_marginals(st["C"], st["space"], st["prior"], ws=st["ws"], marginals=True)
        return edp.scanline_dp(st["C"], st["space"], st["prior"], ws=st["ws"])
    if kind == "windowed":
        from paper_1410_7922_gb300 import proposal
        base = proposal.coarse(st["I0"], st["I1"], st["w"], st["ws_c"])
        centre = proposal.label_centres(base, st["w"]["space"])
        return base, proposal.windowed_edp(st["I0"], st["I1"], st["w"], centre, case["win"], ws=st["ws_w"])
    if kind == "batch":
        edp.solve_batched(st["problems"], st["ws"])
        return [(it["labels"], it["energy4"]) for it in st["items"]]
    if not case["train"]:
        return (edp.net_forward(st["P"], st["x"], st["ws"]),)
    out = edp.net_forward(st["P"], st["x"], st["ws"])
    grad, loss = edp.net_backward(st["P"], out, st["t"], st["ws"])
    # the update works in place: on copies, so that a state can be used again
    P, m, v = st["P"].clone(), st["m"].clone(), st["v"].clone()
    edp.net_adam(P, grad, m, v, ADAM["lr"], ADAM["step"], ADAM["b1"], ADAM["b2"], ADAM["eps"])
    return out, grad, loss, P, m, v


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _edp_work(W, H, Q, R, iters, images, n_img):
    """Bytes: the images or the cost volume in, labels (and energy) out.
    Operations: per pass, label and message one sum (4), a halving and per
    label axis two sweeps (add, min) and a clip; the marginal per solve."""
    N = W * H
    flops = N * Q * (4 * iters * 2 * (5 + 5 * R) + 5)
    if images:
        return {"bytes": n_img * N + 4 * N + 32, "flops": flops + 4 * N * Q}
    return {"bytes": 4 * N * Q + 4 * N, "flops": flops}


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind == "edp":
        Q = case["Q0"] * case["Q1"] * case["Q2"]
        R = sum(q > 1 for q in (case["Q0"], case["Q1"], case["Q2"]))
        return _edp_work(case["W"], case["H"], Q, R, case["iters"], case["images"], 3 if case["Q2"] > 1 else 2)
    if kind == "scanline":
        N, Q = case["W"] * case["H"], case["Q0"]
        if case["marginals"]:
            return {"bytes": 8 * N * Q + 4 * N, "flops": 2 * 6 * N * Q + 3 * N * Q}
        return {"bytes": 4 * N * Q + 4 * N + 8 * case["H"], "flops": 6 * N * Q}
    if kind == "windowed":
        W, H = case["W"], case["H"]
        Qc = (case["Q0"] // 4) * 2 + 1
        a = _edp_work((W + 1) // 2, (H + 1) // 2, Qc * Qc, 2, 1, True, 2)
        b = _edp_work(W, H, case["win"] ** 2, 2, 1, True, 2)
        return {"bytes": 2 * W * H + 8 * W * H, "flops": a["flops"] + b["flops"]}
    if kind == "batch":
        tot = {"bytes": 0, "flops": 0}
        pick = np.random.default_rng(case["mix"])
        for k in range(case["n"]):
            W, H = BATCH_SIZES[int(pick.integers(0, case["max_size"] + 1))]
            if k % 3 == 0:
                Q, R = int(pick.choice([32, 48, 64, 96, 128])), 1
            elif k % 3 == 1:
                Q, R = int(pick.choice([17, 25, 33])) ** 2, 2
            else:
                Q, R = (17 * 17 * 9, 3) if k < 6 else (9 * 9 * 9, 3)
            w = _edp_work(W, H, Q, R, 1, True, 3 if R == 3 else 2)
            tot = {"bytes": tot["bytes"] + w["bytes"], "flops": tot["flops"] + w["flops"]}
        return tot
    npix = case["N"] * case["H"] * case["W"]
    macs = sum(9 * ci * co for ci, co in zip(NET_CHANNELS[:-1], NET_CHANNELS[1:]))
    n_par = macs + sum(NET_CHANNELS[1:])
    if not case["train"]:
        return {"bytes": npix * (5 * 2 + 2 * 4) + 4 * n_par, "flops": 2 * macs * npix}
    first = 9 * NET_CHANNELS[0] * NET_CHANNELS[1]  # no gradient of the features
    # features and targets in, output out; parameters and both moments in and out, gradients out
    return {"bytes": npix * (5 * 2 + 2 * 4 * 2) + 4 * n_par * 7, "flops": 2 * npix * (3 * macs - first)}


# ---------------------------------------------------------------------------
# the same results from plain torch in 64 bits
# ---------------------------------------------------------------------------

def _exact_cost(w: dict, W: int, H: int) -> torch.Tensor:
    """C[y, x, q2, q1, q0] = min(|I1(x + o) - I0(x)| (+ the stereo partner's
    term), cmax); cmax outside the image."""
    s, cmax = w["space"], w["cmax"]
    I0 = torch.as_tensor(w["I0"]).cuda().long()

    def term(I, ox, oy):
        big = torch.full((H, W), -1, dtype=torch.long, device="cuda")
        y0, y1, x0, x1 = max(0, -oy), min(H, H - oy), max(0, -ox), min(W, W - ox)
        if y0 < y1 and x0 < x1:
            big[y0:y1, x0:x1] = (I[y0 + oy:y1 + oy, x0 + ox:x1 + ox] - I0[y0:y1, x0:x1]).abs()
        return big

    Q = s["Q"]
    off = [[s["vmin"][r] + s["step"][r] * q for q in range(Q[r])] for r in range(3)]
    C = torch.empty((H, W, Q[2], Q[1], Q[0]), dtype=torch.long, device="cuda")
    I1 = torch.as_tensor(w["I1"]).cuda().long()
    I2 = None if w["I2"] is None else torch.as_tensor(w["I2"]).cuda().long()
    for q1 in range(Q[1]):
        for q0 in range(Q[0]):
            c1 = term(I1, off[0][q0], off[1][q1] if s["R"] >= 2 else 0)
            if I2 is None:
                C[:, :, 0, q1, q0] = torch.where(c1 < 0, cmax, c1.clamp(max=cmax))
                continue
            for q2 in range(Q[2]):
                c2 = term(I2, off[2][q2], 0)
                C[:, :, q2, q1, q0] = torch.where((c1 < 0) | (c2 < 0), cmax, (c1 + c2).clamp(max=cmax))
    return C


def _min_conv(h: torch.Tensor, prior: dict, lam: torch.Tensor) -> torch.Tensor:
    """min over u of h(u) + V(u, v) on the last three dims of [n, Q2, Q1, Q0];
    lam [n]: the prior weight of each row's edge."""
    g, l1 = prior["g"], prior["l1"]
    cap = g if l1 == 1 else g * g
    per_axis = prior["mode"] == "per_axis"
    lam = lam.view(-1, 1, 1, 1)
    low = h.amin(dim=(1, 2, 3), keepdim=True)
    for d in (3, 2, 1):
        L = h.shape[d]
        if L == 1:
            continue
        o = h.clone()
        for t in range(1, min(g, L)):
            f = t if l1 == 1 else t * t
            a, b = h.narrow(d, 0, L - t) + lam * f, h.narrow(d, t, L - t) + lam * f
            o.narrow(d, t, L - t).copy_(torch.minimum(o.narrow(d, t, L - t), a))
            o.narrow(d, 0, L - t).copy_(torch.minimum(o.narrow(d, 0, L - t), b))
        h = torch.minimum(o, h.amin(dim=d, keepdim=True) + lam * cap) if per_axis else o
    return h if per_axis else torch.minimum(h, low + lam * cap)


def _exact_edp(C: torch.Tensor, prior: dict, iters: int, wh=None, wv=None) -> torch.Tensor:
    """Algorithm 1 with the messages m_k = M(floor(S_k / 2)), one anti-diagonal
    of a pass at a time; labels [H, W]."""
    H, W = C.shape[:2]
    M = [torch.zeros_like(C) for _ in range(4)]  # from +x, -x, +y, -y sweeps
    labels = torch.empty((H, W), dtype=torch.long, device=C.device)
    for it in range(iters):
        for p in range(4):
            incx, incy = p in (0, 2), p < 2
            a, c = (0, 1) if incx else (1, 0)
            b, d = (2, 3) if incy else (3, 2)
            for k in range(W + H - 1):
                r = torch.arange(max(0, k - W + 1), min(H, k + 1), device=C.device)
                y = r if incy else H - 1 - r
                x = (k - r) if incx else W - 1 - (k - r)
                t = C[y, x] + M[a][y, x] + M[b][y, x]
                e = M[d][y, x] - M[c][y, x]
                if it == iters - 1 and p == 3:
                    so = t + M[c][y, x] + M[d][y, x]
                    flat = so.flatten(1)
                    low = flat.amin(dim=1, keepdim=True)
                    labels[y, x] = (flat == low).int().argmax(dim=1)
                for m, s, dx, dy, wt in ((a, t + e, 1 if incx else -1, 0, wh), (b, t - e, 0, 1 if incy else -1, wv)):
                    xn, yn = x + dx, y + dy
                    ok = (xn >= 0) & (xn < W) & (yn >= 0) & (yn < H)
                    if not bool(ok.any()):
                        continue
                    yo, xo = y[ok], x[ok]
                    lam = torch.full_like(yo, prior["lam"])
                    if wt is not None:
                        lam = lam * wt[torch.minimum(yo, yo + dy), torch.minimum(xo, xo + dx)]
                    M[m][yn[ok], xn[ok]] = _min_conv(torch.div(s[ok], 2, rounding_mode="floor"), prior, lam)
    return labels


def _exact_energy(C, labels, space, prior, wh=None, wv=None) -> torch.Tensor:
    H, W = labels.shape
    data = C.flatten(2).gather(2, labels[..., None]).sum()
    Q = space["Q"]
    co = [labels % Q[0], labels // Q[0] % Q[1], labels // (Q[0] * Q[1])]
    cap = prior["g"] if prior["l1"] == 1 else prior["g"] ** 2

    def smooth(u, v):
        f = [(a - b).abs() ** prior["l1"] for a, b in zip(u, v)]
        return sum(t.clamp(max=cap) for t in f) if prior["mode"] == "per_axis" else sum(f).clamp(max=cap)

    h = prior["lam"] * smooth([c[:, :-1] for c in co], [c[:, 1:] for c in co])
    v = prior["lam"] * smooth([c[:-1] for c in co], [c[1:] for c in co])
    if wh is not None:
        h, v = h * wh[:, :-1], v * wv[:-1]
    return torch.stack([data, h.sum(), v.sum(), data + h.sum() + v.sum()])


def _exact_scanline(C: torch.Tensor, prior: dict):
    """Per-row DP over [H, W, Q] with lowest-index ties: labels, row energies."""
    H, W, Q = C.shape
    q = torch.arange(Q, device=C.device)
    d = (q[:, None] - q[None, :]).abs() ** prior["l1"]
    V = prior["lam"] * d.clamp(max=prior["g"] ** prior["l1"])
    S, back = C[:, 0].clone(), []

    def lowest(t):  # values and lowest index over the last dim
        low = t.amin(dim=-1, keepdim=True)
        return low[..., 0], (t == low).int().argmax(dim=-1)

    for x in range(1, W):
        m, arg = lowest(S[:, None, :] + V[None])
        back.append(arg)
        S = C[:, x] + m
    energy, lab = lowest(S)
    out = [lab]
    for arg in reversed(back):
        lab = arg.gather(1, lab[:, None])[:, 0]
        out.append(lab)
    return torch.stack(out[::-1], dim=1), energy


def _exact_marginals(C: torch.Tensor, prior: dict):
    H, W, Q = C.shape

    def chain(Cx):
        S = [Cx[:, 0]]
        lam = torch.full((H,), prior["lam"], device=C.device)
        for x in range(1, W):
            S.append(Cx[:, x] + _min_conv(S[-1][:, None, None], prior, lam)[:, 0, 0])
        return torch.stack(S, dim=1)

    so = chain(C) + chain(C.flip(1)).flip(1) - C
    return (so == so.amin(dim=2, keepdim=True)).int().argmax(dim=2), so


def _exact_net(case: dict, seed: int):
    w = _net_inputs(case, seed)
    P = w["P"].double().cuda().requires_grad_(case["train"])
    h = w["x"].double().cuda().permute(0, 3, 1, 2)
    off = 0
    for k, (ci, co) in enumerate(zip(NET_CHANNELS[:-1], NET_CHANNELS[1:])):
        wt = P[off:off + co * ci * 9].view(co, ci, 3, 3)
        b = P[off + co * ci * 9:off + co * ci * 9 + co]
        off += co * ci * 9 + co
        h = torch.nn.functional.conv2d(h, wt, b, padding=1)
        if k < 5:
            h = torch.relu(h)
    out = h.permute(0, 2, 3, 1)
    if not case["train"]:
        return (out.contiguous(),)
    loss = torch.nn.functional.smooth_l1_loss(out, w["t"].double().cuda())
    loss.backward()
    g = P.grad
    m = ADAM["b1"] * w["m"].double().cuda() + (1 - ADAM["b1"]) * g
    v = ADAM["b2"] * w["v"].double().cuda() + (1 - ADAM["b2"]) * g * g
    c1, c2 = 1 - ADAM["b1"] ** ADAM["step"], 1 - ADAM["b2"] ** ADAM["step"]
    new = P.detach() - ADAM["lr"] * (m / c1) / ((v / c2).sqrt() + ADAM["eps"])
    return out.detach().contiguous(), g, loss.detach().view(1), new, m, v


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind == "net":
        return _exact_net(case, seed)
    if kind == "scanline":
        w = _edp_inputs(case, seed)
        C = _exact_cost(w, case["W"], case["H"]).flatten(2)
        if case["marginals"]:
            return _exact_marginals(C, w["prior"])
        return _exact_scanline(C, w["prior"])
    if kind != "edp":
        return None
    Q = case["Q0"] * case["Q1"] * case["Q2"]
    if case["W"] * case["H"] * Q * case["iters"] > 100_000_000:
        return None  # minutes of work in this form
    w = _edp_inputs(case, seed)
    C = _exact_cost(w, case["W"], case["H"])
    wh = wv = None
    if case["weighted"]:
        I = torch.as_tensor(w["I0"]).cuda().long()
        wh, wv = torch.ones_like(I), torch.ones_like(I)
        wh[:, :-1] += ((I[:, 1:] - I[:, :-1]).abs() < 10).long()
        wv[:-1] += ((I[1:] - I[:-1]).abs() < 10).long()
    labels = _exact_edp(C, w["prior"], case["iters"], wh, wv)
    if not case["images"] and not case["weighted"]:
        return (labels,)
    return labels, _exact_energy(C, labels, w["space"], w["prior"], wh, wv)
