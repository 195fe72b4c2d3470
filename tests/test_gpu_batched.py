"""The batched solve beyond plain parity: problems split between their own
launches and the persistent launch, capture in a CUDA graph with two
replays, and the launch-shape autotuner (every candidate shape gives the
same labels).  Integer results: equal to the oracle bit for bit."""
import numpy as np
import pytest
import torch

from paper_1410_7922_gb300 import autotune
from test_gpu_parity import _batch_items, _oracle_problem, host

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def reset(edp_lib):
    yield
    edp_lib.set_tuning(0, 0, 0)
    edp_lib.set_batch_split(172800)
    edp_lib.set_pass_pairs(edp_lib.PAIRS_AUTO)


def _check(items, iters=1):
    for it in items:
        lab, e = _oracle_problem(it["_w"], iters)
        assert np.array_equal(host(it["labels"]), lab), it["name"]
        assert tuple(int(v) for v in host(it["energy4"])) == e, it["name"]


@pytest.mark.parametrize("split", [0, 1, 1500])
def test_batched_split(edp_lib, split):
    """split 0: every problem in the persistent launch; 1: every problem on
    its own launches; 1500 pixels: the larger ones on their own."""
    edp_lib.set_batch_split(split)
    items = _batch_items(edp_lib, n=9)
    probs = edp_lib.make_problems(items)
    ws = torch.empty(edp_lib.batch_workspace_size(probs), dtype=torch.uint8, device="cuda")
    edp_lib.solve_batched(probs, ws)
    torch.cuda.synchronize()
    assert edp_lib.get_device_status(ws) == 0
    _check(items)


def test_batched_graph_capture_and_replay(edp_lib):
    """One uncaptured call (sets the kernels' attributes), a capture, then
    two replays with the outputs cleared in between."""
    edp_lib.set_batch_split(1500)
    items = _batch_items(edp_lib, n=9)
    probs = edp_lib.make_problems(items)
    ws = torch.empty(edp_lib.batch_workspace_size(probs), dtype=torch.uint8, device="cuda")
    edp_lib.solve_batched(probs, ws)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        with torch.cuda.graph(g, stream=st):
            edp_lib.solve_batched(probs, ws, stream=st)
    torch.cuda.current_stream().wait_stream(st)
    for _ in range(2):
        for it in items:
            it["labels"].fill_(-1)
            it["energy4"].fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        assert edp_lib.get_device_status(ws) == 0
        _check(items)


def test_batched_autotune_candidates_agree(edp_lib):
    """autotune.tune times every (rows per block, warps per row) candidate;
    each candidate's labels are the same, and equal to the oracle's."""
    items = _batch_items(edp_lib, n=6)
    probs = edp_lib.make_problems(items)
    ws = torch.empty(edp_lib.batch_workspace_size(probs), dtype=torch.uint8, device="cuda")
    results = []

    def run():
        for it in items:
            it["labels"].fill_(-1)
        edp_lib.solve_batched(probs, ws)
        torch.cuda.synchronize()
        results.append([it["labels"].clone() for it in items])

    r, w, ms, table = autotune.tune(run, rows=(0, 1, 2), warps=(0, 2, 4), reps=1)
    assert len(table) >= 2 and ms > 0
    for res in results[1:]:
        assert all(torch.equal(a, b) for a, b in zip(results[0], res))
    _check(items)


def _random_items(edp_lib, shapes):
    """Problems of random images: (W, H, label axes) each."""
    rng = np.random.default_rng(len(shapes))
    items = []
    for W, H, Q in shapes:
        space = {"R": len(Q), "Q": tuple(Q), "vmin": tuple(-(q // 2) for q in Q), "step": (1,) * len(Q)}
        w = dict(name=f"{W}x{H} {Q}", I2=None, space=space, l2=1, cmax=20, cost_mode="pair",
                 prior={"lam": 5, "g": 3, "l1": 1, "mode": "per_axis"})
        w["I0"], w["I1"] = (rng.integers(0, 256, size=(H, W)).astype(np.uint8) for _ in range(2))
        items.append(dict(w, I0=torch.from_numpy(w["I0"]).cuda(), I1=torch.from_numpy(w["I1"]).cuda(), iters=1, _w=w,
                          labels=torch.zeros((H, W), dtype=torch.int32, device="cuda"),
                          energy4=torch.empty(4, dtype=torch.int64, device="cuda")))
    return items


@pytest.mark.parametrize("shapes,whole", [
    ([(50, 40, (21, 13)), (50, 40, (5, 4))], True),        # every problem on its own launches
    ([(50, 40, (21, 13)), (40, 30, (16,))], True),         # a shared launch after one of them
    ([(50, 40, (21, 13)), (40, 30, (16,))], False),        # the same in two waves
])
def test_batched_status_word(edp_lib, shapes, whole):
    """The status word of a batch covers the problems that run on their own
    launches: 0 after a good call on a workspace full of ones, EDP_ERR_TIMEOUT
    after one whose first row band waited in vain, whatever ran after it."""
    items = _random_items(edp_lib, shapes)
    probs = edp_lib.make_problems(items)
    n = edp_lib.batch_workspace_size(probs if whole else edp_lib.make_problems(items[:1]))
    ws = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")
    for hold in (0, 1, 0):
        try:
            edp_lib.set_spin_limit(20000 if hold else 0)
            edp_lib.test_hold_band(hold)
            edp_lib.solve_batched(probs, ws)
            assert edp_lib.get_device_status(ws) == (edp_lib.ERR_TIMEOUT if hold else 0)
        finally:
            edp_lib.test_hold_band(0)
            edp_lib.set_spin_limit(0)
        if not hold:
            _check(items)


@pytest.mark.parametrize("split,alone", [(172800, True), (172801, False), (76800, False), (12001, False), (12000, True),
                                         (0, False)])
def test_batch_split_holds_for_multi_axis_problems(edp_lib, split, alone):
    """A 120x100 problem of 9 x 9 labels runs by itself at the default setting
    and where the setting says so, else in the shared launch (which leaves the
    name of the last solve's kernel as it was)."""
    items = _random_items(edp_lib, [(120, 100, (9, 9))])
    probs = edp_lib.make_problems(items)
    ws = torch.empty(edp_lib.batch_workspace_size(probs), dtype=torch.uint8, device="cuda")
    edp_lib.set_tuning(0, 0, 3)
    edp_lib.solve(torch.zeros((4, 4, 81), dtype=torch.int32, device="cuda"), items[0]["space"], items[0]["prior"])
    edp_lib.set_tuning(0, 0, 0)
    assert edp_lib.last_pass_kernel() == "edp_pass_team_kernel"
    edp_lib.set_batch_split(split)
    edp_lib.solve_batched(probs, ws)
    assert edp_lib.last_pass_kernel() == ("edp_pass_line2_kernel" if alone else "edp_pass_team_kernel")
    assert edp_lib.get_device_status(ws) == 0
    _check(items)
