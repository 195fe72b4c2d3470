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
