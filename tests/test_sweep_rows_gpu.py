"""The sweep's row classes and its way from a push to a pull, against the
one-kernel-per-phase path on the same chain: rows of one link, at and beside
the length a warp pushes with others (64), at and beside the length a block
pushes (512) and far beyond it (cut into pieces that all blocks share), more
rows of 65 to 512 links than a block's queue holds (1024), and moves that
reach the pull limit right after moves far below it (the dense moved cash is
then set from the lists). FP64: the two paths differ by the order of the
additions only, n eps of the largest value at most."""
import numpy as np
import pytest

from paper_2008_02710_gb300 import synth

pytestmark = pytest.mark.gpu

LENS = [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 511, 512, 513, 1023, 1025, 5000]


def _chain(n, lens, weighted, seed):
    rng = np.random.default_rng(seed)
    deg = np.full(n, 3, dtype=np.int64)
    deg[rng.choice(n, len(lens), replace=False)] = lens
    row_ptr = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    col = rng.integers(0, n, row_ptr[-1]).astype(np.int32)
    col[row_ptr[:-1]] = (np.arange(n) + 1) % n  # one cycle through all nodes
    w = (rng.integers(1, 1 << 20, row_ptr[-1]) * 2.0 ** -20).astype(np.float32) if weighted else None
    return synth.CSR(n, row_ptr, col, w)


def _masks(n, shares, seed):
    rng = np.random.default_rng(seed)
    return np.stack([(rng.random(n) < s).astype(np.uint8) for s in shares])


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n,lens", [(33, [64, 65]), (4097, LENS), (70001, LENS * 3), (3000, [100] * 1500)])
def test_row_classes_and_surprise_pulls(n, lens, weighted):
    from paper_2008_02710_gb300.rlgl import Chain
    csr = _chain(n, lens, weighted, seed=n)
    masks = _masks(n, [0.1, 0.95, 0.9, 0.2, 0.0, 1.0, 0.05], seed=1)
    out = []
    for persistent in (1, 0):
        with Chain(csr) as ch:
            ch.set_params(persistent=persistent, pull_crossover=0.6)
            ch.set_masks(masks)
            info = ch.solve("mask", tol=0.0, max_steps=20, raise_on_noconv=False)
            assert info["moves"] == 20 and ch.get_params().persistent == persistent
            out.append((*ch.get_state(), ch.move_log(20), info))
    (ca, ha, la, ia), (cb, hb, lb, ib) = out
    assert [r["mode"] for r in la] == [r["mode"] for r in lb]
    assert [r["green"] for r in la] == [r["green"] for r in lb]
    assert [r["edges_pushed"] for r in la] == [r["edges_pushed"] for r in lb]
    assert {r["mode"] for r in la} >= {0, 1, 2}
    eps = 20 * (max(lens) + n / 100 + 64) * 2.0 ** -53
    assert np.abs(ha - hb).max() <= eps * np.abs(hb).max()
    assert np.abs(ca - cb).max() <= eps * np.abs(hb).max()


@pytest.mark.parametrize("r", [2, 3])
@pytest.mark.parametrize("theta_lag", [0, 1])
def test_exponents_of_the_threshold(r, theta_lag):
    """theta = (sum v^r / N)^(1/r) for the exponents with their own code: the
    logged threshold of the first move is that of the state it starts from."""
    from paper_2008_02710_gb300.rlgl import Chain
    csr = _chain(5003, LENS, False, seed=3)
    with Chain(csr) as ch:
        c, _ = ch.get_state()
        ch.set_params(r=r, theta_lag=theta_lag, theta_scale=0.5)
        ch.solve("link_threshold", tol=0.0, max_steps=3, raise_on_noconv=False)
        log = ch.move_log(3)
    v = np.abs(c) / np.diff(csr.row_ptr)
    want = 0.5 * np.mean(v ** r) ** (1.0 / r)
    assert abs(log[0]["theta"] - want) <= 1e-12 * want
    if theta_lag:
        assert log[1]["theta"] == log[0]["theta"]
