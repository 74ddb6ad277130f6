"""The compaction of the contraction's table: coarse rows that end on, cross
and fill the warps' runs of 2,048 slots, against numpy."""
import numpy as np
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2608_01503_gb300 as lc  # noqa: E402

N, M = 6000, 60_000


def regular(n, k):
    """Every vertex joined to its k nearest on either side of a ring."""
    v = np.repeat(np.arange(n), k)
    return gg.from_edges(n, v, (v + np.tile(np.arange(1, k + 1), n)) % n, seed=2, wmin=1, wmax=9)


def random(n, m):
    rng = np.random.default_rng(1)
    s, t = rng.integers(0, n, m), rng.integers(0, n, m)
    return gg.from_edges(n, s[s != t], t[s != t], seed=1, wmin=1, wmax=9)


LABELS = {
    "two": lambda n: np.arange(n) % 2,                     # rows of many runs
    "singletons": lambda n: np.arange(n),                  # rows far below a run
    "64 each": lambda n: np.arange(n) // 64,               # a row per run on the regular graph
    "63 each": lambda n: np.arange(n) // 63,
    "half and singletons": lambda n: np.maximum(np.arange(n) - n // 2, 0),
    "random": lambda n: np.unique(np.random.default_rng(3).integers(0, 700, n), return_inverse=True)[1],
    "one": lambda n: np.zeros(n, np.int64),                # nothing leaves the cluster
}


@pytest.mark.parametrize("labels", list(LABELS))
@pytest.mark.parametrize("graph", ["regular", "random"])
def test_contraction_equals_numpy(graph, labels):
    rp, col, ew = regular(N, 8) if graph == "regular" else random(N, M)
    lab = LABELS[labels](N).astype(np.int32)
    nc = int(lab.max()) + 1
    src, dst = lab[np.repeat(np.arange(N), np.diff(rp))].astype(np.int64), lab[col].astype(np.int64)
    out = src != dst
    key, inv = np.unique(src[out] * nc + dst[out], return_inverse=True)
    want = np.bincount(inv, weights=ew[out], minlength=key.size).astype(np.int64) if key.size else np.zeros(0, np.int64)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    crp, ccol, cew, cvw = (t.cpu().numpy() for t in lc.lc_contract(dev(rp), dev(col), dev(ew), dev(np.ones(N, np.int64)),
                                                                  dev(lab), nc)[:4])
    got = np.repeat(np.arange(nc), np.diff(crp)) * nc + ccol[: crp[-1]]
    order = np.argsort(got)
    assert np.array_equal(got[order], key) and np.array_equal(cew[: crp[-1]][order], want)
    assert np.array_equal(cvw, np.bincount(lab, minlength=nc))
