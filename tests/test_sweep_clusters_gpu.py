"""Green nodes and long rows that lie together by id, as a host's pages, a
block-round-robin range or ids sorted by degree do: the same moves as the
one-kernel-per-phase path, and a move that takes no longer than one whose
green nodes are spread over the ids."""
import numpy as np
import pytest

from paper_2008_02710_gb300 import synth

pytestmark = pytest.mark.gpu


def _chain(n, deg, seed):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.as_tensor(deg, device="cuda"), 0)
    col = torch.randint(0, n, (int(row_ptr[-1]),), generator=gen, device="cuda", dtype=torch.int32)
    col[row_ptr[:-1]] = ((torch.arange(n, device="cuda") + 1) % n).to(torch.int32)  # one cycle through all nodes
    return synth.CSR(n, row_ptr, col, None)


def _eighths(n):
    masks = np.zeros((8, n), dtype=np.uint8)
    for k in range(8):
        masks[k, k * n // 8:(k + 1) * n // 8] = 1
    return masks


# Groups of 32, 64 (FP64) and 128 (MIXED) nodes, the last one ragged; the
# third chain has more rows of 65 to 512 links in a block than its queue for
# them holds (1024), whatever block they fall to: 250000 rows over the SMs.
@pytest.mark.parametrize("precision,n,long_rows", [("fp64", 5003, 700), ("fp64", 330017, 3000), ("fp64", 330017, 250000),
                                                   ("mixed", 330017, 3000), ("mixed", 1300003, 3000)])
def test_clustered_moves(precision, n, long_rows):
    import torch
    from paper_2008_02710_gb300.rlgl import Chain
    if long_rows == 250000:
        assert long_rows // torch.cuda.get_device_properties(0).multi_processor_count > 1024
    deg = np.full(n, 3, dtype=np.int64)
    deg[:long_rows] = 80
    csr = _chain(n, deg, seed=n)
    moves, out = 16, []
    for persistent in (1, 0):
        with Chain(csr, precision=precision) as ch:
            ch.set_params(persistent=persistent, pull_crossover=2.0)  # pushes only
            ch.set_masks(_eighths(n))
            ch.solve("mask", tol=0.0, max_steps=moves, raise_on_noconv=False)
            out.append((*ch.get_state(), ch.move_log(moves)))
    (ca, ha, la), (cb, hb, lb) = out
    assert [(r["green"], r["edges_pushed"], r["mode"]) for r in la] == [(r["green"], r["edges_pushed"], r["mode"]) for r in lb]
    # the two differ by the order of the additions alone: at most a rounding
    # for each of a node's additions a move (in-links: 3 or 80 a row, at random)
    in_links = int(torch.bincount(csr.col).max())
    eps = moves * (in_links + 64) * (2.0 ** -53 if precision == "fp64" else 2.0 ** -24)
    scale = np.abs(hb).max()
    assert np.abs(ha - hb).max() <= eps * scale
    assert np.abs(ca - cb).max() <= eps * scale


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_clustered_moves_take_no_longer(precision):
    """An eighth of the nodes, together or every eighth (R-MAT with ids at
    random: as many links). On one SM in eight the former took 2.0 times the
    latter; 1.4 leaves room for a busy machine."""
    from paper_2008_02710_gb300.rlgl import Chain
    n = 1 << 20
    together = _eighths(n)
    spread = np.ascontiguousarray(together.reshape(8, 8, n // 8).transpose(0, 2, 1).reshape(8, n))
    us = []
    with Chain(synth.rmat_chain_n_device(n, 16, 3), precision=precision) as ch:
        for masks in (together, spread):
            ch.set_masks(masks)
            best = []
            for _ in range(5):
                ch.reset(None)
                ch.solve("mask", tol=0.0, max_steps=24, raise_on_noconv=False)
                best.append(np.median([sum(r["phase_us"][2:]) for r in ch.move_log(24)[8:]]))
            us.append(min(best))
    assert us[0] <= 1.4 * us[1], us
