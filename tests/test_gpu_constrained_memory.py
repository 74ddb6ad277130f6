"""What a constrained level takes for its filtered graph goes back before the
next level."""
import ctypes

import numpy as np
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2608_01503_gb300 as lc  # noqa: E402


def test_filtered_graph_is_returned_before_the_next_level():
    g = gg.modularity_inputs(*gg.rmat_csr(14, seed=2))  # hubs, several levels
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (g.row_ptr, g.col, g.ew, g.vw)]
    classes = (torch.arange(g.n, device="cuda") % 3).to(torch.int32)
    labels, res = torch.zeros(g.n, dtype=torch.int32, device="cuda"), lc._Result()
    held, taken, log = {}, [], []

    def alloc(_ctx, nbytes, _stream):
        x = torch.empty(max(1, nbytes), dtype=torch.uint8, device="cuda")
        held[x.data_ptr()] = (x, len(taken))
        taken.append(nbytes)
        log.append(("take", len(taken) - 1))
        return x.data_ptr()

    def dealloc(_ctx, ptr, _nbytes, _stream):
        log.append(("give", held.pop(ptr)[1]))

    c = lc._c_opts(lc.Options(allocator="library"), lc._stream_handle())
    c.alloc, c.dealloc = fns = lc._AllocFn(alloc), lc._FreeFn(dealloc)
    csr = lc._Csr(g.n, g.nnz, t[0].data_ptr(), t[1].data_ptr())
    rc = lc.load().lc_cluster_constrained(ctypes.byref(csr), t[3].data_ptr(), t[2].data_ptr(), g.lam_num, g.lam_den,
                                          classes.data_ptr(), ctypes.byref(c), labels.data_ptr(), ctypes.byref(res))
    torch.cuda.synchronize()
    assert rc == 0 and not held and res.levels > 2 and fns
    # the records of the full and of the filtered level 0: 32 bytes a vertex
    records = [i for i, b in enumerate(taken) if b == 32 * g.n]
    assert len(records) == 2
    given = log.index(("give", records[1]))
    # everything taken from the filtered row offsets to its records' end of use
    # is back before the next level's dense ids are taken
    first = max(i for i in range(records[1]) if taken[i] == 8 * (g.n + 1))
    nxt = next(k for k, (what, i) in enumerate(log) if what == "take" and i > records[1] and taken[i] == 4 * g.n)
    assert given < nxt
    back = {i for what, i in log[:nxt] if what == "give"}
    kept = [i for i in range(first, log[nxt][1]) if i not in back and taken[i] != 32]  # 32: the level's own parameters
    assert kept == [], [(i, taken[i]) for i in kept]
