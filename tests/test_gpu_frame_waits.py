"""The bounded waits of the split line kernel's frame (one-axis rows, split
lines, label boxes), made to run out without any fault: the test hook
edp_test_hold_band makes one band wait for hand-off data no producer
publishes.  Every kernel of the solve returns, the status word says
EDP_ERR_TIMEOUT, and the next solve on the same workspace is exact."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_parity import dev, host, reset_tuning, sp  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limit", [1000, 20000])
@pytest.mark.parametrize("Q", [(16,), (27, 15), (21, 13), (5, 5, 5)])
def test_records_of_a_paired_sweep_run_out(edp_lib, Q, limit):
    """Twice as many blocks as bands: those of the second half wait for rows
    of the first half that the held band never completes, all lanes of the
    polling warp together."""
    rng = np.random.default_rng(sum(Q))
    H, W = 24, 20
    C = rng.integers(0, 21, size=(H, W, int(np.prod(Q)))).astype(np.int32)
    prior = {"lam": 5, "g": 3, "l1": 1, "mode": "joint"}
    want = oracle.edp(C, sp(Q), prior)
    gC, ws = dev(C), edp_lib.workspace(edp_lib.OP_SOLVE, W, H, sp(Q), prior, 1)
    edp_lib.set_tuning(1, 0, 0)
    edp_lib.set_pass_pairs(True)
    for band in (1, 5, 23):
        try:
            edp_lib.set_spin_limit(limit)
            edp_lib.test_hold_band(band)
            edp_lib.solve(gC, sp(Q), prior, ws=ws)
            assert edp_lib.get_device_status(ws) == edp_lib.ERR_TIMEOUT
        finally:
            edp_lib.test_hold_band(0)
            edp_lib.set_spin_limit(0)
        got = host(edp_lib.solve(gC, sp(Q), prior, ws=ws))
        assert edp_lib.get_device_status(ws) == 0
        assert np.array_equal(got, want), band


@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("Q,W,rows", [((16,), 200, 0), ((64,), 90, 2), ((37,), 60, 1), ((1,), 50, 0), ((21, 13), 12, 2)])
def test_bands_with_a_whole_row_of_records_do_not_wait_for_those_below(edp_lib, Q, W, rows, pairs):
    """A band whose consumer never takes a column still runs to its end (in the
    second pass of a pair: the band above that), long before the held one
    gives up: a solve advances with any number of running blocks."""
    rng = np.random.default_rng(W)
    H, hold = 40, 4
    C = rng.integers(0, 21, size=(H, W, int(np.prod(Q)))).astype(np.int32)
    prior = {"lam": 5, "g": 3, "l1": 1, "mode": "joint"}
    ws = edp_lib.workspace(edp_lib.OP_SOLVE, W, H, sp(Q), prior, 1)
    edp_lib.set_tuning(rows, 0, 0)
    edp_lib.set_pass_pairs(pairs)
    gC = dev(C)
    edp_lib.solve(gC, sp(Q), prior, ws=ws)  # (the kernel is loaded before the timed launch)
    trace = torch.zeros((H, 4), dtype=torch.int64, device="cuda")  # of the first launch
    try:
        edp_lib.set_trace(trace)
        edp_lib.set_spin_limit(200000)
        edp_lib.test_hold_band(hold)
        edp_lib.solve(gC, sp(Q), prior, ws=ws)
        assert edp_lib.get_device_status(ws) == edp_lib.ERR_TIMEOUT
    finally:
        edp_lib.test_hold_band(0)
        edp_lib.set_spin_limit(0)
        edp_lib.set_trace(None)
    t = host(trace)
    start, end = t[0, 0], t[:, 1]
    free = hold - 1 if pairs else hold  # bands that end by themselves
    assert (t[:hold + 1, 1] > 0).all()
    assert end[:free].max() - start < (end[hold] - start) / 2, (end[:hold + 1] - start)


def test_solves_at_once_on_several_streams(edp_lib):
    """One-axis, two-axis and windowed solves in flight together, the one-axis
    ones on streams of both priorities: labels as when each runs alone."""
    rng = np.random.default_rng(6)
    jobs = []

    def job(Q, W, H, win=0, priority=0):
        space, prior = sp(Q), {"lam": 8, "g": 3, "l1": 1, "mode": "per_axis"}
        C = dev(rng.integers(0, 21, size=(H, W, win * win if win else int(np.prod(Q)))).astype(np.int32))
        st = torch.cuda.Stream(priority=priority)
        if win:
            centre = dev((rng.integers(0, 3, size=(H, W, 2)) + 10).astype(np.int32))
            ws = edp_lib.workspace_windowed(W, H, space, prior, win, 1)
            run = lambda lab, s: edp_lib.solve_windowed(C, centre, win, space, prior, ws=ws, labels=lab, stream=s)
        else:
            ws = edp_lib.workspace(edp_lib.OP_SOLVE, W, H, space, prior, 1)
            run = lambda lab, s: edp_lib.solve(C, space, prior, ws=ws, labels=lab, stream=s)
        want = torch.empty((H, W), dtype=torch.int32, device="cuda")
        run(want, None)
        jobs.append((run, ws, st, want, torch.empty_like(want)))

    for priority in (0, -1, 0):
        job((64,), 300, 375, priority=priority)
    job((33, 33), 60, 240)
    job((27, 15), 80, 265)
    job((33, 33), 90, 480, win=9)
    torch.cuda.synchronize()
    for _ in range(3):
        for run, ws, st, want, got in jobs:
            with torch.cuda.stream(st):
                got.fill_(-1)
            run(got, st)
    torch.cuda.synchronize()
    for run, ws, st, want, got in jobs:
        assert edp_lib.get_device_status(ws) == 0
        assert torch.equal(got, want)


@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("Q,win,l1", [((13, 13), 5, 1), ((20, 20), 9, 1), ((33, 40), 15, 1), ((13, 13), 5, 2),
                                      ((40,), 7, 1)])
def test_windowed_waits_run_out(edp_lib, Q, win, l1, pairs):
    """Label boxes of two axes on the frame's rows, the other windowed forms on
    the multi-axis kernel."""
    rng = np.random.default_rng(win + l1)
    H, W, R = 40, 17, len(Q)
    centre = np.stack([rng.integers(-2, q + 2, size=(H, W)) for q in Q], axis=-1).astype(np.int32)
    Cw = rng.integers(0, 31, size=(H, W, win ** R)).astype(np.int32)
    prior = {"lam": 4, "g": 3, "l1": l1, "mode": "per_axis"}
    want = oracle.edp_windowed(Cw, centre, sp(Q), prior, win, iters=1)
    ws = edp_lib.workspace_windowed(W, H, sp(Q), prior, win, 1)
    gC, gc = dev(Cw), dev(centre)
    edp_lib.set_pass_pairs(pairs)
    edp_lib.set_tuning(2, 0, 0)
    for band in (1, 6):
        try:
            edp_lib.set_spin_limit(2000)
            edp_lib.test_hold_band(band)
            edp_lib.solve_windowed(gC, gc, win, sp(Q), prior, ws=ws)
            assert edp_lib.get_device_status(ws) == edp_lib.ERR_TIMEOUT
        finally:
            edp_lib.test_hold_band(0)
            edp_lib.set_spin_limit(0)
        got = edp_lib.solve_windowed(gC, gc, win, sp(Q), prior, ws=ws)
        assert edp_lib.get_device_status(ws) == 0
        assert np.array_equal(host(got), want), band
    assert edp_lib.last_pass_kernel() == ("edp_pass_line2_kernel" if R == 2 and l1 == 1 else "edp_pass_team_kernel")


@pytest.mark.parametrize("pairs", [0, 1])
@pytest.mark.parametrize("Q", [(16,), (200,), (9, 9), (33, 33), (65, 65), (11, 7, 5), (9, 9, 9), (17, 17, 9)])
def test_waits_of_the_default_kernels_run_out(edp_lib, Q, pairs):
    """The kernels the planner picks: records up to 512 labels, copies above."""
    rng = np.random.default_rng(sum(Q))
    H, W = (20, 8) if np.prod(Q) > 2000 else (36, 20)
    C = rng.integers(0, 21, size=(H, W, int(np.prod(Q)))).astype(np.int32)
    prior = {"lam": 5, "g": 3, "l1": 1, "mode": "per_axis"}
    gC, ws = dev(C), edp_lib.workspace(edp_lib.OP_SOLVE, W, H, sp(Q), prior, 1)
    edp_lib.set_pass_pairs(pairs)
    try:
        edp_lib.set_spin_limit(20000)
        edp_lib.test_hold_band(2)
        edp_lib.solve(gC, sp(Q), prior, ws=ws)
        assert edp_lib.get_device_status(ws) == edp_lib.ERR_TIMEOUT
    finally:
        edp_lib.test_hold_band(0)
        edp_lib.set_spin_limit(0)
    got = host(edp_lib.solve(gC, sp(Q), prior, ws=ws))
    assert edp_lib.get_device_status(ws) == 0
    assert edp_lib.last_pass_kernel() == "edp_pass_line2_kernel"
    assert np.array_equal(got, oracle.edp(C, sp(Q), prior, tier=1))


def test_more_bands_than_blocks(edp_lib):
    """Tall frames of one row per block: rings shorter than a row between bands
    that run one after another, label boxes and split lines."""
    rng = np.random.default_rng(5)
    H, W, Q = 6000, 12, (13, 11)
    prior = {"lam": 4, "g": 3, "l1": 1, "mode": "per_axis"}
    centre = np.stack([rng.integers(-2, q + 2, size=(H, W)) for q in Q], axis=-1).astype(np.int32)
    Cw = rng.integers(0, 31, size=(H, W, 25)).astype(np.int32)
    C = rng.integers(0, 21, size=(H, W, 143)).astype(np.int32)
    want_w = oracle.edp_windowed(Cw, centre, sp(Q), prior, 5, iters=1)
    want = oracle.edp(C, sp(Q), prior, tier=1)
    edp_lib.set_tuning(1, 0, 0)
    for pairs in (0, 1, 2):
        edp_lib.set_pass_pairs(pairs)
        assert np.array_equal(host(edp_lib.solve_windowed(dev(Cw), dev(centre), 5, sp(Q), prior, iters=1)), want_w), pairs
        assert np.array_equal(host(edp_lib.solve(dev(C), sp(Q), prior)), want), pairs
