"""The source order of the in-link copy (the nodes with the most out-links
first, kept in shared memory by the all-green sweep) at its edges: more long
rows than fit, rows of equal length that do not all fit, more rows of the
longest class (4095 links and more) than fit, long rows last, first and in
between. Step 0 against numpy, all-green moves and the invariant residual
against the one-kernel-per-phase path."""
import numpy as np
import pytest

from paper_2008_02710_gb300 import synth

pytestmark = pytest.mark.gpu

CAP = {"fp64": 4096, "mixed": 14336}  # sources the sweep keeps


def _degrees(kind, cap, rng):
    n = 4 * cap
    deg = rng.integers(2, 9, n)
    some = cap + cap // 2
    if kind == "cap binds":        # a whole length more would not fit
        deg[rng.choice(n, some, replace=False)] = rng.integers(64, 90, some)
    elif kind == "ties":           # one length, more rows than fit: none is kept
        deg[rng.choice(n, some, replace=False)] = 80
    elif kind == "last":           # every kept source has to move to the front
        deg[-(cap // 2):] = rng.integers(64, 200, cap // 2)
    elif kind == "first":          # none has to
        deg[:cap // 2] = rng.integers(64, 200, cap // 2)
    elif kind == "none":
        pass
    elif kind == "one":
        deg[n // 2] = 5000
    return deg


def _chain(deg, rng):
    n = len(deg)
    row_ptr = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    col = rng.integers(0, n, row_ptr[-1]).astype(np.int32)
    col[row_ptr[:-1]] = (np.arange(n) + 1) % n  # one cycle through all nodes
    return synth.CSR(n, row_ptr, col, None)


def _check(csr, precision):
    import torch
    from paper_2008_02710_gb300.rlgl import Chain
    dev = synth.CSR(csr.n, torch.from_numpy(csr.row_ptr).cuda(), torch.from_numpy(csr.col).cuda(), None)
    deg = np.diff(csr.row_ptr)
    in_links = np.bincount(csr.col, minlength=csr.n)
    moves, out = 6, []
    for persistent in (1, 0):
        with Chain(dev, precision=precision) as ch:
            ch.set_params(persistent=persistent)
            c0, h0 = ch.get_state()
            # C_0 = M_0 P - M_0, one rounding an in-link and three more
            src = np.repeat(h0 / deg, deg)
            want = np.bincount(csr.col, weights=src, minlength=csr.n) - h0
            eps = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
            bound = (in_links + 3) * 2.0 ** -53 * (np.bincount(csr.col, weights=src, minlength=csr.n) + h0) + eps * np.abs(want)
            assert (np.abs(c0 - want) <= bound).all()
            ch.solve("all_green", tol=0.0, max_steps=moves, raise_on_noconv=False)
            out.append((*ch.get_state(), ch.invariant_residual()))
    (ca, ha, ra), (cb, hb, rb) = out
    tol = moves * (in_links.max() + 8) * (2.0 ** -53 if precision == "fp64" else 2.0 ** -24)
    assert np.abs(ha - hb).max() <= tol * np.abs(hb).max()
    assert np.abs(ca - cb).max() <= tol * np.abs(hb).max()
    assert ra <= tol and rb <= tol


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", ["cap binds", "ties", "last", "first", "none", "one"])
def test_source_order(kind, precision):
    rng = np.random.default_rng(7)
    _check(_chain(_degrees(kind, CAP[precision], rng), rng), precision)


def test_more_of_the_longest_rows_than_fit():
    rng = np.random.default_rng(8)
    n = 5000
    deg = np.full(n, 3)
    deg[rng.choice(n, 4200, replace=False)] = rng.integers(4095, 4200, 4200)
    _check(_chain(deg, rng), "fp64")
