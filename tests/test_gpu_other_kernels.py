"""The scan-pass kernels beside the split line kernel's frame, which serve what
it does not: the warp-per-row kernel (one label axis, costs off a 16-byte
boundary) and the multi-axis kernel (general_kernel = 3, the lane-group form
at 2).  Label counts around their lane cuts, rows per block, both pass
schedules, more bands than blocks, per-edge weights, waits that run out.
Integer results: equal to the oracle bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_parity import dev, host, reset_tuning, sp  # noqa: F401

pytestmark = pytest.mark.gpu

R1, TEAM = "edp_pass_r1_kernel", "edp_pass_team_kernel"


def off4(C):
    """The cost volume on the device, 4 bytes off a 16-byte boundary."""
    buf = torch.zeros(C.size + 1, dtype=torch.int32, device="cuda")
    view = buf[1:].view(C.shape)
    view.copy_(dev(C))
    return view


@pytest.mark.parametrize("Q", [1, 5, 16, 31, 32, 33, 64, 100, 129, 256])
@pytest.mark.parametrize("g", [1, 2, 4, 9, 300])
def test_warp_per_row(edp_lib, Q, g):
    rng = np.random.default_rng(Q * 1000 + g)
    C = rng.integers(0, 21, size=(19, 27, Q)).astype(np.int32)
    prior = {"lam": int(rng.integers(1, 25)), "g": g, "l1": 1, "mode": "joint"}
    got = host(edp_lib.solve(off4(C), sp((Q,)), prior, iters=2))
    assert edp_lib.last_pass_kernel() == R1
    assert np.array_equal(got, oracle.edp(C, sp((Q,)), prior, iters=2, tier=1))


@pytest.mark.parametrize("rows", [2, 3, 5, 8, 16])
@pytest.mark.parametrize("pairs", [False, True])
def test_warp_per_row_rows_per_block(edp_lib, rows, pairs):
    rng = np.random.default_rng(rows)
    C = rng.integers(0, 21, size=(37, 41, 64)).astype(np.int32)
    prior = {"lam": 20, "g": 4, "l1": 1, "mode": "joint"}
    edp_lib.set_tuning(rows, 0, 0)
    edp_lib.set_pass_pairs(pairs)
    got = host(edp_lib.solve(off4(C), sp((64,)), prior, iters=2))
    assert edp_lib.last_pass_kernel() == R1
    assert edp_lib.last_pass_launches() == (4 if pairs else 8)
    assert np.array_equal(got, oracle.edp(C, sp((64,)), prior, iters=2, tier=1))


@pytest.mark.parametrize("Q,l1", [(7, 1), (64, 1), (256, 1), (16, 2), (64, 2)])
def test_warp_per_row_weighted(edp_lib, Q, l1):
    rng = np.random.default_rng(Q + l1)
    H, W = 19, 23
    C = rng.integers(0, 21, size=(H, W, Q)).astype(np.int32)
    wh, wv = (rng.integers(0, 4, size=(H, W)).astype(np.uint8) for _ in range(2))
    prior = {"lam": 3, "g": 4, "l1": l1, "mode": "joint"}
    got = host(edp_lib.solve_weighted(off4(C), sp((Q,)), prior, dev(wh), dev(wv), 3, iters=2))
    assert edp_lib.last_pass_kernel() == R1
    assert np.array_equal(got, oracle.edp_weighted(C, sp((Q,)), prior, wh, wv, iters=2))


@pytest.mark.parametrize("mode", ["joint", "per_axis"])
@pytest.mark.parametrize("general", [2, 3])
@pytest.mark.parametrize("Q", [(5, 4), (9, 9), (17, 9), (21, 13), (27, 15), (33, 33), (9, 9, 9), (17, 17, 9), (5, 4, 3)])
def test_multi_axis_kernel(edp_lib, Q, general, mode):
    rng = np.random.default_rng(sum(Q) + general)
    n = int(np.prod(Q))
    H, W = (9, 7) if n > 500 else (17, 21)
    C = rng.integers(0, 21, size=(H, W, n)).astype(np.int32)
    prior = {"lam": int(rng.integers(1, 12)), "g": int(rng.integers(1, 5)), "l1": 1, "mode": mode}
    want = oracle.edp(C, sp(Q), prior, iters=2, tier=1)
    for rows in (0, 2):
        edp_lib.set_tuning(rows, 0, general)
        got = host(edp_lib.solve(dev(C), sp(Q), prior, iters=2))
        assert edp_lib.last_pass_kernel() == TEAM
        assert np.array_equal(got, want), rows


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("Q", [(16,), (5, 4), (9, 9)])
def test_more_bands_than_blocks(edp_lib, mode, Q):
    rng = np.random.default_rng(sum(Q) + mode)
    C = rng.integers(0, 21, size=(12000, 3, int(np.prod(Q)))).astype(np.int32)
    prior = {"lam": int(rng.integers(1, 12)), "g": 3, "l1": 1, "mode": "per_axis" if len(Q) > 1 else "joint"}
    edp_lib.set_pass_pairs(mode)
    edp_lib.set_tuning(2, 0, 0 if len(Q) == 1 else 3)
    got = host(edp_lib.solve(off4(C) if len(Q) == 1 else dev(C), sp(Q), prior, iters=2))
    assert edp_lib.last_pass_kernel() == (R1 if len(Q) == 1 else TEAM)
    assert np.array_equal(got, oracle.edp(C, sp(Q), prior, iters=2, tier=1))


@pytest.mark.parametrize("pairs", [0, 1])
@pytest.mark.parametrize("Q,general", [((16,), 0), ((9, 9), 3), ((17, 17, 9), 3), ((21, 13), 2)])
def test_waits_run_out(edp_lib, Q, general, pairs):
    rng = np.random.default_rng(sum(Q))
    H, W = 36, 20
    C = rng.integers(0, 21, size=(H, W, int(np.prod(Q)))).astype(np.int32)
    prior = {"lam": 5, "g": 3, "l1": 1, "mode": "per_axis" if len(Q) > 1 else "joint"}
    gC, ws = (off4 if len(Q) == 1 else dev)(C), edp_lib.workspace(edp_lib.OP_SOLVE, W, H, sp(Q), prior, 1)
    edp_lib.set_tuning(2, 0, general)
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
    assert edp_lib.last_pass_kernel() == (R1 if len(Q) == 1 else TEAM)
    assert np.array_equal(got, oracle.edp(C, sp(Q), prior, tier=1))
