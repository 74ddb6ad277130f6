"""No edge is read before row_ptr is known to end at the caller's count: a
count beyond the arrays is refused like any other bad argument."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2608_01503_gb300 as lc  # noqa: E402

N = 1000


def ring():
    v = torch.arange(N, dtype=torch.int64, device="cuda")
    col = torch.sort(torch.stack(((v - 1) % N, (v + 1) % N), 1), 1).values.flatten().to(torch.int32)
    return (torch.arange(0, 2 * N + 1, 2, dtype=torch.int64, device="cuda"), col,
            torch.ones(2 * N, dtype=torch.int32, device="cuda"), torch.ones(N, dtype=torch.int64, device="cuda"))


def test_columns_longer_than_the_weights():
    """A column buffer with room to spare beside exact weights."""
    rp, col, ew, vw = ring()
    room = torch.zeros(1 << 26, dtype=torch.int32, device="cuda")
    room[: col.numel()] = col
    lab = torch.zeros(N, dtype=torch.int32, device="cuda")
    for call in (lambda c: lc.lc_cluster(rp, c, ew, vw, 1, 50), lambda c: lc.lc_cluster_leiden(rp, c, ew, vw, 1, 50),
                 lambda c: lc.lc_local_move(rp, c, ew, vw, 1, 50, lab.clone()),
                 lambda c: lc.lc_objective(rp, c, ew, vw, 1, 50, lab),
                 lambda c: lc.lc_cluster(rp, c, ew, vw, 1, 50, opts=lc.Options(validate=False))):
        with pytest.raises(lc.LCError) as e:
            call(room)
        assert e.value.code == 1
        call(col)  # the count itself is fine
    torch.cuda.synchronize()


@pytest.mark.parametrize("nnz", [2 * N - 1, 2 * N + 1, 1 << 24, 1 << 36, 1 << 41, 1 << 62])
def test_count_beyond_the_arrays(nnz):
    rp, col, ew, vw = ring()
    lab, res = torch.zeros(N, dtype=torch.int32, device="cuda"), lc._Result()
    csr = lc._Csr(N, nnz, rp.data_ptr(), col.data_ptr())
    c = lc._c_opts(lc.Options(), lc._stream_handle())
    rc = lc.load().lc_cluster(ctypes.byref(csr), vw.data_ptr(), ew.data_ptr(), 1, 50, ctypes.byref(c), lab.data_ptr(),
                              ctypes.byref(res))
    torch.cuda.synchronize()
    assert rc == 1
