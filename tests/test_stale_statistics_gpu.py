"""The stale threshold's statistics, gathered by a move's selection from the
cash before it: the third move's theta is (sum v^r / N)^(1/r) of the cash that
one move leaves, for the exponents with their own code and both thresholds."""
import numpy as np
import pytest

from paper_2008_02710_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("schedule", ["threshold", "link_threshold"])
@pytest.mark.parametrize("r", [1, 2, 3, 5])
@pytest.mark.parametrize("n", [4097, 330017])  # groups of 32 and 64 nodes
def test_statistics_of_a_move(n, r, schedule):
    from paper_2008_02710_gb300.rlgl import Chain
    csr = synth.rmat_chain_n_device(n, 8, 11)
    deg = np.diff(csr.row_ptr.cpu().numpy())
    with Chain(csr) as ch:
        ch.set_params(r=r, theta_lag=1, theta_scale=0.5)
        ch.solve(schedule, tol=0.0, max_steps=1, raise_on_noconv=False)
        c, _ = ch.get_state()
        ch.reset(None)
        ch.solve(schedule, tol=0.0, max_steps=3, raise_on_noconv=False)
        log = ch.move_log(3)
    v = np.abs(c) / (deg if schedule == "link_threshold" else 1)
    want = 0.5 * np.mean(v ** r) ** (1.0 / r)
    # sums of n terms in FP64, and the order of the additions to the cash
    assert abs(log[2]["theta"] - want) <= 1e-11 * want
    assert log[1]["theta"] == log[0]["theta"]
