"""The edge checks name the row of a fault wherever it lies: dense rows, rows
that end on the check's step and run boundaries, and entries with thousands of
empty rows between them; unaligned arrays take the scalar loads."""
import gc

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2608_01503_gb300 as lc  # noqa: E402

SHAPES = {
    "dense": lambda rng: np.full(700, 40),
    "steps": lambda rng: rng.choice([0, 1, 31, 32, 33, 127, 128, 129, 1023, 1024, 1025], 1200),
    "sparse": lambda rng: np.where(rng.random(300_000) < 0.004, rng.integers(1, 9, 300_000), 0),
    "mixed": lambda rng: np.concatenate((np.full(300, 50), np.zeros(70_000, np.int64), rng.integers(0, 3, 5000))),
}


def graph(name, offset):
    """Rows of the shape's lengths with valid, sorted, loop-free columns (not
    symmetric), on the device; offset: entries by which col and ew are
    shifted in memory."""
    rng = np.random.default_rng(5)
    deg = SHAPES[name](rng).astype(np.int64)
    n = deg.size
    rp = np.concatenate(([0], np.cumsum(deg)))
    col = np.concatenate([np.sort(rng.choice(n - 1, d, replace=False)) + 0 for d in deg if d] or [np.zeros(0)])
    row = np.repeat(np.arange(n), deg)
    col = (col + (col >= row)).astype(np.int32)  # skip the row itself
    return rp, col, np.ones(col.size, np.int32), row


def check(rp, col, ew, offset):
    def shifted(a):
        t = torch.empty(a.size + offset, dtype=torch.int32, device="cuda")
        t[offset:] = torch.from_numpy(a).cuda()
        return t[offset:]

    with pytest.raises(lc.LCError) as e:
        lc.lc_cluster(torch.from_numpy(rp).cuda(), shifted(col), shifted(ew),
                      torch.ones(rp.size - 1, dtype=torch.int64, device="cuda"), 1, 2)
    return e.value.code, e.value.detail


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("name", list(SHAPES))
def test_fault_is_reported_with_its_row(name, offset):
    rp, col, ew, row = graph(name, offset)
    assert check(rp, col, ew, offset)[0] == 2  # only the symmetry fails
    rng = np.random.default_rng(9)
    first = np.zeros(col.size, bool)
    first[rp[:-1][np.diff(rp) > 0]] = True
    places = list(rng.integers(0, col.size, 3)) + [0, col.size - 1]
    for at in places:
        bad = col.copy()
        bad[at] = row[at]
        code, detail = check(rp, bad, ew, offset)
        assert (code, detail) == (3, row[at])  # self-loop
        bad[at] = rp.size - 1
        assert check(rp, bad, ew, offset) == (1, row[at])  # column out of range
        w = ew.copy()
        w[at] = 0
        assert check(rp, col, w, offset) == (5, row[at])  # weight
        if not first[at]:
            bad = col.copy()
            bad[at] = bad[at - 1]
            assert check(rp, bad, ew, offset) == (4, row[at])  # duplicate


@pytest.mark.parametrize("limit,code_ok", [(0, 0), (100_000, 7)])
def test_faults_of_the_graph_and_labels_come_before_memory(limit, code_ok):
    """Scratch is taken while the graph is still being read: a self-loop is
    reported before bad labels, both before a scratch limit that is too low,
    and the device holds what it held before."""
    n = 4000
    rp = np.arange(0, 2 * n + 2, 2)
    ring = np.stack(((np.arange(n) - 1) % n, (np.arange(n) + 1) % n), 1)
    col = np.sort(ring, 1).astype(np.int32).ravel()
    loop = col.copy()
    loop[2 * 700] = 700  # row 700: {699, 701} -> {700, 701}
    good, bad = np.zeros(n, np.int32), np.full(n, n, np.int32)

    def code(c, labels):
        a = [torch.from_numpy(x).cuda() for x in (rp, c, np.ones(2 * n, np.int32), np.ones(n, np.int64))]
        lab = torch.from_numpy(labels).cuda()
        gc.collect()  # what earlier tests left must not be freed in between
        base = torch.cuda.memory_allocated()
        try:
            lc.lc_local_move(*a, 1, 2, lab, opts=lc.Options(scratch_limit=limit))
            got = 0
        except lc.LCError as e:
            got = e.code
        assert torch.cuda.memory_allocated() == base
        return got

    assert code(loop, bad) == 3 and code(col, bad) == 1 and code(loop, good) == 3
    assert code(col, good) == code_ok
