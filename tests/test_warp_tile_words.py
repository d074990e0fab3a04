"""With FP32 cash the all-green sweep keeps a row's in-link sum in the shared
word of the row's end (no GPU). Restated here: which words the 32 lanes of a
warp read and write between the barrier before the merge loop and the one
after it. A word that one lane writes must be no other lane's to read or
write; a read of the next row's end after a lane's last item (its row may lie
whole in the next lane, which writes its sum) breaks that."""
import os
import re

import numpy as np
import pytest

from tests.test_warp_tiles import partition, rows_of

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_02710_gb300", "csrc",
                   "rlgl_power.cuh")


def _words(ends, start0, ne, ipt, guarded):
    """Per lane the words (rows; nr: the word past the last) it reads and writes in the merge loop."""
    nr = len(ends)
    ends = list(ends) + [1 << 30]
    reads, writes = [set() for _ in range(32)], [set() for _ in range(32)]
    total = nr + ne
    for lane in range(32):
        d = lane * ipt
        if d >= total:
            continue
        i = next(k for k in range(max(0, d - ne), min(d, nr) + 1) if k >= min(d, nr) or ends[k] >= d - k)
        j = d - i
        whole = j == (start0 if i == 0 else ends[i - 1])  # (read before the barrier)
        end = ends[i]
        reads[lane].add(i)
        for q in range(ipt):
            if d + q >= total:
                break
            if j < end:
                j += 1
                continue
            if whole:
                writes[lane].add(i)
            i += 1
            whole = True
            if not guarded or q + 1 < ipt:
                end = ends[i]
                reads[lane].add(i)
    return reads, writes


def _clashes(deg, ipt, guarded):
    t_ptr = rows_of(deg)
    tr, te = partition(t_ptr, 32 * ipt)
    n = 0
    for b in range(len(tr) - 1):
        r0, e0, r1, e1 = tr[b], te[b], tr[b + 1], te[b + 1]
        if r1 == r0:
            continue  # (every item a link of one row: no merge)
        reads, writes = _words(t_ptr[r0 + 1:r1 + 1] - e0, t_ptr[r0] - e0, e1 - e0, ipt, guarded)
        for a in range(32):
            for c in range(32):
                if a != c:
                    n += len(writes[a] & (reads[c] | writes[c]))
    return n


@pytest.mark.parametrize("seed", [1, 2])
def test_no_lane_reads_a_word_that_another_writes(seed):
    rng = np.random.default_rng(seed)
    deg = np.minimum(rng.zipf(1.7, 4000), 900)
    deg[rng.choice(4000, 500, replace=False)] = 0
    assert _clashes(deg, 12, guarded=True) == 0
    assert _clashes(deg, 12, guarded=False) > 0  # (the model sees it)


def test_the_loop_has_the_guard_and_the_barrier():
    src = open(SRC).read()
    loop = src[src.index("struct PowWarp"):src.index("power_split_rows")]
    assert re.search(r"if \(q \+ 1 < kPowIpt\) end = ws\.ends\[i\];", loop)
    assert re.search(r"__syncwarp\(\);\s+const T run = warp_segscan", loop)
    assert "reinterpret_cast<T*>(ends)" not in src
