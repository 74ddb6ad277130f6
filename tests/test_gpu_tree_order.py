"""pLeidenR's order of the trees: small forests are ranked by counting, a
forest with a very large tree is radix-sorted; both against the oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2608_01503_gb300 as lc  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# a star's tree holds about half of its leaves: 20,000 leaves stay below 2^30
# pairs, 120,000 do not
@pytest.mark.parametrize("leaves", [1, 31, 2_000, 20_000, 120_000])
def test_star(leaves):
    rp, col, ew = gg.from_edges(leaves + 1, np.zeros(leaves, np.int64), np.arange(1, leaves + 1))
    g = gg.cpm_inputs(rp, col, ew, 1, 4 * leaves + 4)
    labels, res = lc.lc_cluster_leiden(dev(rp), dev(col), dev(ew), dev(g.vw), g.lam_num, g.lam_den)
    ref, orc, _ = oracle.pleiden(g)
    assert np.array_equal(labels.cpu().numpy(), ref) and res["phi"] == orc["phi"]


@pytest.mark.parametrize("degrees", [[7, 8, 9, 15, 16, 17, 31, 32, 33], [255, 256, 257, 511, 513, 1023, 1025],
                                     [4095, 4096, 4097, 9000]])
def test_rows_around_the_group_sizes(degrees):
    """Rows where the refinement's walks change from a thread to 16 lanes, a
    warp, 128 and 512 threads: stars of these degrees whose leaves and centres
    are joined at random."""
    rng = np.random.default_rng(len(degrees))
    n, at, src, dst = len(degrees) + sum(degrees), len(degrees), [], []
    for k, d in enumerate(degrees):
        src.append(np.full(d, k))
        dst.append(np.arange(at, at + d))
        at += d
    m = 2 * n
    src.append(rng.integers(0, n, m))
    dst.append(rng.integers(0, n, m))
    s, t = np.concatenate(src), np.concatenate(dst)
    rp, col, ew = gg.from_edges(n, s[s != t], t[s != t], seed=3, wmin=1, wmax=5)
    for g in (gg.modularity_inputs(rp, col, ew), gg.cpm_inputs(rp, col, ew, 1, 50)):
        labels, res = lc.lc_cluster_leiden(dev(rp), dev(col), dev(ew), dev(g.vw), g.lam_num, g.lam_den)
        ref, orc, _ = oracle.pleiden(g)
        assert np.array_equal(labels.cpu().numpy(), ref) and res["phi"] == orc["phi"]
