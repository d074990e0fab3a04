"""The sweep's statistics are sums in a fixed order: the first move of a solve
takes its threshold from the same cash in every run, so that it must log the
same ||C||_1 and theta. The blocks' FP64 sums meet in FP64 additions in any
order, at most one a block: they may differ by as many roundings of 2^-53."""
import numpy as np
import pytest

from paper_2008_02710_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("schedule", ["threshold", "link_threshold"])
@pytest.mark.parametrize("n", [4099, 300007, 1300001])  # a group a warp, some, and groups of 128 nodes
def test_one_cash_has_one_sum(n, schedule):
    import torch
    from paper_2008_02710_gb300.rlgl import Chain
    blocks = torch.cuda.get_device_properties(0).multi_processor_count
    got = []
    with Chain(synth.rmat_chain_n_device(n, 8, 5), precision="mixed") as ch:
        for _ in range(12):
            ch.reset(None)
            ch.solve(schedule, tol=0.0, max_steps=1, raise_on_noconv=False)
            r = ch.move_log(1)[0]
            got.append((r["l1_cash"], r["theta"]))
    got = np.array(got)
    spread = (got.max(axis=0) - got.min(axis=0)) / got.max(axis=0)
    assert (spread <= (blocks + 2) * 2.0 ** -53).all(), spread
