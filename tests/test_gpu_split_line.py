"""The split line kernel's frame at the sizes where its cuts, its rings and its
dispatch can go wrong: label lines at the edges of the segment cuts, one label
axis at the edges of the lane cuts, label boxes of every odd side, many bands
on a small chip's worth of blocks, per-edge weights, misaligned costs (other
kernels), the scanline DP's lane cuts and pieces.  Integer results: equal to
the oracle bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_parity import dev, host, reset_tuning, sp  # noqa: F401

pytestmark = pytest.mark.gpu


def _prior(rng, mode="joint", l1=1):
    return {"lam": int(rng.integers(0, 9)), "g": int(rng.integers(1, 7)), "l1": l1, "mode": mode}


@pytest.mark.parametrize("mode", ["joint", "per_axis"])
@pytest.mark.parametrize("Q", [(2, 2), (1, 9), (9, 1), (11, 7), (20, 12), (21, 13), (27, 15), (31, 19), (33, 33),
                               (40, 33), (64, 8), (65, 40), (72, 72), (11, 7, 5), (1, 1, 6), (9, 9, 9), (16, 16, 3)])
def test_multi_axis_cuts(edp_lib, Q, mode):
    rng = np.random.default_rng(sum(Q) + len(mode))
    n = int(np.prod(Q))
    H, W = (5, 9) if n > 1000 else (14, 11)
    for hi, g in ((21, 3), (3, 1), (200, max(Q) + 2)):  # far truncation: every segment boundary is crossed
        C = rng.integers(0, hi, size=(H, W, n)).astype(np.int32)
        prior = {"lam": int(rng.integers(0, 9)), "g": g, "l1": 1, "mode": mode}
        want = oracle.edp(C, sp(Q), prior, iters=2)
        for rows in (0, 1, 3):
            edp_lib.set_tuning(rows, 0, 0)
            got = host(edp_lib.solve(dev(C), sp(Q), prior, iters=2))
            assert np.array_equal(got, want), (prior, rows, edp_lib.last_pass_kernel())


@pytest.mark.parametrize("H,W", [(1, 1), (1, 30), (30, 1), (2, 3), (61, 5), (5, 61)])
@pytest.mark.parametrize("Q", [(21, 13), (5, 5, 5), (37,)])
def test_frames(edp_lib, Q, H, W):
    """Degenerate frames, and tall ones on one row per block (many hand-offs)."""
    rng = np.random.default_rng(H * 64 + W)
    C = rng.integers(0, 21, size=(H, W, int(np.prod(Q)))).astype(np.int32)
    prior = _prior(rng)
    want = oracle.edp(C, sp(Q), prior, iters=2)
    for rows, pairs in ((0, edp_lib.PAIRS_AUTO), (1, True), (1, False), (4, True)):
        edp_lib.set_tuning(rows, 0, 0)
        edp_lib.set_pass_pairs(pairs)
        assert np.array_equal(host(edp_lib.solve(dev(C), sp(Q), prior, iters=2)), want), (rows, pairs)


@pytest.mark.parametrize("l1", [1, 2])
@pytest.mark.parametrize("Q", [1, 2, 15, 16, 31, 32, 33, 63, 64, 65, 127, 128, 129, 254, 255, 256])
def test_one_axis_cuts(edp_lib, Q, l1):
    rng = np.random.default_rng(Q * 2 + l1)
    H, W = 11, 17
    C = rng.integers(0, 40, size=(H, W, Q)).astype(np.int32)
    wh, wv = (rng.integers(0, 4, size=(H, W)).astype(np.uint8) for _ in range(2))
    for g in (1, 4, 40):
        prior = {"lam": 3, "g": g, "l1": l1, "mode": "joint"}
        if l1 == 2 and g == 40:
            continue
        want = oracle.edp(C, sp((Q,)), prior, iters=2)
        wantw = oracle.edp_weighted(C, sp((Q,)), prior, wh, wv, iters=2)
        for rows in (0, 1, 3):
            edp_lib.set_tuning(rows, 0, 0)
            assert np.array_equal(host(edp_lib.solve(dev(C), sp((Q,)), prior, iters=2)), want), (g, rows)
        edp_lib.set_tuning(0, 0, 0)
        assert np.array_equal(host(edp_lib.solve_weighted(dev(C), sp((Q,)), prior, dev(wh), dev(wv), 3, iters=2)), wantw)


@pytest.mark.parametrize("Q", [(37,), (9, 9), (21, 13)])
def test_misaligned_costs(edp_lib, Q):
    """A cost volume 4 bytes off a 16-byte boundary gives the same labels."""
    rng = np.random.default_rng(sum(Q))
    n = int(np.prod(Q))
    C = rng.integers(0, 21, size=(9, 12, n)).astype(np.int32)
    prior = _prior(rng)
    buf = torch.zeros(C.size + 1, dtype=torch.int32, device="cuda")
    view = buf[1:].view(C.shape)
    view.copy_(dev(C))
    assert np.array_equal(host(edp_lib.solve(view, sp(Q), prior)), oracle.edp(C, sp(Q), prior))


@pytest.mark.parametrize("mode", ["joint", "per_axis"])
@pytest.mark.parametrize("win", [3, 5, 7, 9, 11, 13, 15])
def test_windowed_boxes(edp_lib, win, mode):
    """Boxes that overlap, lie far apart and are clamped at the space's ends."""
    rng = np.random.default_rng(win)
    Q, H, W = (33, 40), 13, 10
    prior = {"lam": 4, "g": 3, "l1": 1, "mode": mode}
    for spread in (2, 60):
        centre = (rng.integers(-spread, spread + 1, size=(H, W, 2)) + 16).astype(np.int32)
        Cw = rng.integers(0, 31, size=(H, W, win * win)).astype(np.int32)
        want = oracle.edp_windowed(Cw, centre, sp(Q), prior, win, iters=2)
        for rows in (0, 1, 3):
            edp_lib.set_tuning(rows, 0, 0)
            got = host(edp_lib.solve_windowed(dev(Cw), dev(centre), win, sp(Q), prior, iters=2))
            assert np.array_equal(got, want), (spread, rows)


@pytest.mark.parametrize("Q", [1, 2, 5, 63, 64, 65, 127, 128, 129, 255, 256])
@pytest.mark.parametrize("W", [1, 2, 15, 16, 17, 66, 300])
def test_scanline_one_axis(edp_lib, Q, W):
    """Lane cuts (64, 128, 256 labels), the cost ring's depth, pieces of
    back-pointers that start anywhere, heavy ties."""
    rng = np.random.default_rng(Q * 512 + W)
    for hi, lam, g in ((3, 1, 2), (60, 3, 5), (9, 0, 3), (250, 1, 300)):
        C = rng.integers(0, hi, size=(5, W, Q)).astype(np.int32)
        prior = {"lam": lam, "g": g, "l1": 1, "mode": "joint"}
        lab, row_e = oracle.scanline_dp(C, sp((Q,)), prior, tier=1)
        glab, grow = edp_lib.scanline_dp(dev(C), sp((Q,)), prior)
        assert np.array_equal(host(glab), lab) and np.array_equal(host(grow), row_e), prior
        mlab, marg = edp_lib.scanline_marginals(dev(C), sp((Q,)), prior, marginals=True)
        edp_lib.set_tuning(2, 0, 0)  # the general kernel
        olab, omarg = edp_lib.scanline_marginals(dev(C), sp((Q,)), prior, marginals=True)
        glab, grow = edp_lib.scanline_dp(dev(C), sp((Q,)), prior)
        edp_lib.set_tuning(0, 0, 0)
        assert torch.equal(mlab, olab) and torch.equal(marg, omarg)
        assert np.array_equal(host(glab), lab) and np.array_equal(host(grow), row_e), prior


@pytest.mark.parametrize("split", [0, 1500, 172800])
def test_batch_sizes_around_the_split(edp_lib, split):
    """Two-axis problems just below and at the sizes from which they run by
    themselves, beside one-axis ones, under three settings of the split."""
    rng = np.random.default_rng(3)
    items = []
    for W, H, Q in ((49, 40, (5, 4)), (50, 40, (5, 4)), (119, 100, (9, 9)), (120, 100, (9, 9)), (60, 50, (16,))):
        w = dict(name=f"{W}x{H} {Q}", I2=None, space=sp(Q, [-(q // 2) for q in Q], [1] * len(Q)),
                 prior={"lam": 5, "g": 3, "l1": 1, "mode": "per_axis"}, l2=1, cmax=20, cost_mode="pair")
        w["I0"], w["I1"] = (rng.integers(0, 256, size=(H, W)).astype(np.uint8) for _ in range(2))
        items.append(dict(w, I0=dev(w["I0"]), I1=dev(w["I1"]), iters=1, _w=w,
                          labels=torch.empty((H, W), dtype=torch.int32, device="cuda"),
                          energy4=torch.empty(4, dtype=torch.int64, device="cuda")))
    probs = edp_lib.make_problems(items)
    ws = torch.empty(edp_lib.batch_workspace_size(probs), dtype=torch.uint8, device="cuda")
    edp_lib.set_batch_split(split)
    try:
        edp_lib.solve_batched(probs, ws)
    finally:
        edp_lib.set_batch_split(172800)
    torch.cuda.synchronize()
    for it in items:
        w = it["_w"]
        C = oracle.cost_volume(w["I0"], w["I1"], None, w["space"], 1, 20)
        lab = oracle.edp(C, w["space"], w["prior"])
        assert np.array_equal(host(it["labels"]), lab), it["name"]
        assert tuple(int(v) for v in host(it["energy4"])) == oracle.energy(C, lab, w["space"], w["prior"]), it["name"]


@pytest.mark.parametrize("Q,step", [((33, 5), (1, 1)), ((40,), (-1, 1)), ((65, 9), (-1, 1)), ((32, 33), (1, -1))])
@pytest.mark.parametrize("l2", [1, 2])
def test_pair_cost_inside_and_border(edp_lib, Q, step, l2):
    """Frames with pixels whose whole label window lies inside the image."""
    rng = np.random.default_rng(sum(Q) + l2)
    space = sp(Q, [-(q // 2) * s for q, s in zip(Q, step)], step[:len(Q)])
    I0, I1 = (rng.integers(0, 256, size=(43, 90)).astype(np.uint8) for _ in range(2))
    got = edp_lib.cost_volume(dev(I0), dev(I1), None, space, l2, 300)
    assert np.array_equal(host(got), oracle.cost_volume(I0, I1, None, space, l2, 300))


def test_net_gradient_of_many_tiles_per_block(edp_lib):
    """The gradients of four images are the mean of the single ones' (the
    output gradients scale by a power of two, exact in bfloat16), so only the
    order of float32 sums differs: 1e-3 of each tensor's largest entry."""
    rng = np.random.default_rng(8)
    N, H, W = 4, 240, 321
    P = torch.from_numpy(rng.normal(0, 0.08, size=edp_lib.net_param_count()).astype(np.float32)).cuda()
    x = torch.from_numpy(rng.uniform(-1, 1, size=(N, H, W, 5)).astype(np.float32)).bfloat16().cuda()
    t = torch.from_numpy(rng.normal(0, 3, size=(N, H, W, 2)).astype(np.float32)).cuda()

    def grad(a, b):
        ws = edp_lib.net_workspace(b - a, H, W)
        xs, ts = x[a:b].contiguous(), t[a:b].contiguous()
        g, _ = edp_lib.net_backward(P, edp_lib.net_forward(P, xs, ws), ts, ws)
        return g.double().cpu().numpy()

    got, want = grad(0, N), sum(grad(i, i + 1) for i in range(N)) / N
    chan = [5, 32, 32, 32, 32, 32, 2]
    o = 0
    for ci, co in zip(chan[:-1], chan[1:]):
        for n in (co * ci * 9, co):
            assert np.abs(got[o:o + n] - want[o:o + n]).max() <= 1e-3 * np.abs(want[o:o + n]).max(), (ci, co, n)
            o += n


@pytest.mark.parametrize("Q", [(33, 33), (21, 13), (9, 9), (65, 65), (40, 1), (20, 3)])
def test_fused_cost_switch_of_every_space(edp_lib, Q):
    """Images to labels and energy with the fused pair cost asked for: spaces
    whose kernel has no such build get their cost volume as ever."""
    rng = np.random.default_rng(sum(Q))
    H, W = 14, 20
    I0, I1 = (rng.integers(0, 256, size=(H, W)).astype(np.uint8) for _ in range(2))
    space, prior = sp(Q, [-(q // 2) for q in Q], [1, 1]), {"lam": 4, "g": 3, "l1": 1, "mode": "per_axis"}
    C = oracle.cost_volume(I0, I1, None, space, 1, 20)
    want = oracle.edp(C, space, prior)
    for shape in ((0, 0), (1, 12)):  # the planner's, and one that may need another build
        try:
            edp_lib.set_fused_cost(True)
            edp_lib.set_tuning(shape[0], 0, 0, warps_per_row=shape[1])
            lab, e = edp_lib.solve_images(dev(I0), dev(I1), None, space, prior, 1, 20)
        finally:
            edp_lib.set_fused_cost(False)
            edp_lib.set_tuning(0, 0, 0)
        assert np.array_equal(host(lab), want), shape
        assert tuple(int(v) for v in host(e)) == oracle.energy(C, want, space, prior), shape


def test_fused_cost_switch_and_coarse_labels(edp_lib):
    """The coarse level of a 65 x 65 space has 33 x 33 labels."""
    rng = np.random.default_rng(4)
    I0, I1 = (dev(rng.integers(0, 256, size=(46, 60)).astype(np.uint8)) for _ in range(2))
    space = sp((65, 65), (-32, -32), (1, 1))
    prior = {"lam": 4, "g": 3, "l1": 1, "mode": "per_axis"}
    want = edp_lib.coarse_labels(I0, I1, space, prior, 1, 20)
    try:
        edp_lib.set_fused_cost(True)
        got = edp_lib.coarse_labels(I0, I1, space, prior, 1, 20)
    finally:
        edp_lib.set_fused_cost(False)
    assert torch.equal(got, want)


@pytest.mark.parametrize("far", [2 ** 31 - 11, 2 ** 31 - 1, -2 ** 31 + 5, -2 ** 31])
@pytest.mark.parametrize("step", [1, -1])
def test_pair_cost_far_displacements(edp_lib, far, step):
    """Displacements at the ends of int32, where a window's end wraps when
    added up in 32 bits: every label lies outside the image and costs cmax."""
    H, W = 20, 90
    I0, I1 = (torch.zeros((H, W), dtype=torch.uint8, device="cuda") for _ in range(2))
    for Q, vmin in (((40,), [far]), ((40, 6), [far, 0]), ((40, 6), [0, far]), ((40, 6), [far, far])):
        space = sp(Q, vmin, [step] * len(Q))
        assert bool((edp_lib.cost_volume(I0, I1, None, space, 1, 7) == 7).all()), (Q, vmin)


@pytest.mark.parametrize("Q,rows,warps,kernel", [
    ((33, 33), 0, 12, "edp_pass_line2_kernel"), ((33, 33), 8, 12, "edp_pass_line2_kernel"),  # one row fits
    ((33, 33), 30, 0, "edp_pass_line2_kernel"), ((65, 65), 4, 0, "edp_pass_line2_kernel"),
    ((17, 17, 9), 0, 8, "edp_pass_line2_kernel"),
    ((17, 17, 9), 0, 9, "edp_pass_team_kernel"),  # 384 threads hold 8 compute and 4 copy warps
    ((17, 17, 9), 2, 12, "edp_pass_team_kernel"),
])
def test_pinned_launch_shapes(edp_lib, Q, rows, warps, kernel):
    """A pinned number of warps is never dropped: a kernel that can run it
    does; pinned rows are an upper bound."""
    rng = np.random.default_rng(rows + warps)
    C = rng.integers(0, 21, size=(9, 6, int(np.prod(Q)))).astype(np.int32)
    prior = {"lam": 4, "g": 3, "l1": 1, "mode": "per_axis"}
    edp_lib.set_tuning(rows, 0, 0, warps_per_row=warps)
    got = host(edp_lib.solve(dev(C), sp(Q), prior))
    assert edp_lib.last_pass_kernel() == kernel
    assert np.array_equal(got, oracle.edp(C, sp(Q), prior))
