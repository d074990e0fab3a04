"""Beyond L2 an FP32 chain's green rows are pushed in about the order of the
nodes, whatever their length: the order decides how the cash is rounded. Two
targets receive 0.5 from one of the first nodes and many amounts of 2^-27 from
rows spread over all nodes; each of those is lost if it comes after the 0.5
(half a unit of its last place is 2^-25) and kept if it comes before."""
import numpy as np
import pytest

from paper_2008_02710_gb300 import synth

pytestmark = pytest.mark.gpu

N = 6_600_000          # beyond 96 MB of cash, 1/d and history
TINY = 2.0 ** -27


def test_rows_in_the_order_of_the_nodes():
    import torch
    from paper_2008_02710_gb300.rlgl import Chain
    deg = np.full(N, 2, dtype=np.int64)
    long_rows = np.arange(400, N, 330)       # cut into pieces
    short_rows = np.arange(450, N, 100)
    deg[long_rows] = 600
    deg[0] = 100                             # a row between the two classes
    short_rows = short_rows[(deg[short_rows] == 2) & (short_rows < N - 1)]
    c = np.zeros(N)
    to_a, to_b = 100, 200                    # targets (their rows carry nothing)
    row_ptr = np.concatenate([[0], np.cumsum(deg)])
    rng = np.random.default_rng(1)
    col = rng.integers(300, N, row_ptr[-1]).astype(np.int32)
    col[row_ptr[:-1]] = (np.arange(N) + 1) % N   # one cycle through all nodes
    # a: 0.5 from the row of 100 links, the small amounts from rows of 2
    col[row_ptr[0] + 1] = to_a
    c[0] = 0.5 * 100
    col[row_ptr[short_rows] + 1] = to_a
    c[short_rows] = TINY * 2
    # b: 0.5 from a row of 2, the small amounts from rows of 600
    col[row_ptr[2] + 1] = to_b
    c[2] = 0.5 * 2
    col[row_ptr[long_rows] + 1] = to_b
    c[long_rows] = TINY * 600
    c[N - 1] = -c.sum()                      # (cash sums to zero; this row feeds neither)
    csr = synth.CSR(N, torch.from_numpy(row_ptr).cuda(), torch.from_numpy(col).cuda(), None)
    with Chain(csr, c=c, h=np.full(N, 1.0 / N), precision="mixed") as ch:
        ch.set_params(pull_crossover=2.0, refresh_factor=0.0, stall_moves=0)
        ch.set_masks(np.ones((1, N), dtype=np.uint8))
        ch.solve("mask", tol=0.0, max_steps=1, raise_on_noconv=False)
        assert ch.move_log(1)[0]["mode"] == 1 and ch.move_log(1)[0]["green"] == N
        got, _ = ch.get_state()
    kept_a = (got[to_a] - 0.5) / (TINY * len(short_rows))
    kept_b = (got[to_b] - 0.5) / (TINY * len(long_rows))
    assert 0.0 <= kept_a <= 0.4 and 0.0 <= kept_b <= 0.4, (kept_a, kept_b)
