"""The degree bins are built while row_ptr is still being checked: whatever
row_ptr holds, the phase that counts the bins and the phase that places the
vertices agree, and the call is refused with the first faulty row."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2608_01503_gb300 import _build

MAX_DEG = np.array([8, 16, 32, 128, 256, 512, 1024, 2048, 4096], np.int32)


def row_pointers():
    rng = np.random.default_rng(3)
    i64 = np.iinfo(np.int64)
    return {
        "sound": np.concatenate(([0], np.cumsum(rng.integers(0, 6000, 4000)))),
        "falling": np.concatenate((-3 * 10 ** 9 * np.arange(1000), [5000])),
        "up and back": np.array([0, 1 << 30, 1 << 31, 3 << 30, 0]),
        "around 32 bits": np.cumsum(np.concatenate(([0], rng.choice([0, 7, 5000, (1 << 31) - 1, 1 << 31, (1 << 32) + 5,
                                                                      -((1 << 32) - 5000), -7], 3000)))),
        "anything": np.concatenate(([0], rng.integers(i64.min, i64.max, 5000), [77])),
        "ends of 64 bits": np.concatenate(([0], np.tile([i64.max, i64.min, 0, -1], 500), [9])),
    }


@pytest.fixture(scope="module")
def bins(tmp_path_factory):
    """The two phases' bins of every row, by the library's own header."""
    d = tmp_path_factory.mktemp("bin_rule")
    src = d / "shim.cpp"
    src.write_text('#include "lc_bin_rule.cuh"\n'
                   'extern "C" void bins(const int64_t *rp, int64_t n, const int32_t *max_deg, int32_t *deg, int32_t *bin) {\n'
                   '  for (int64_t v = 0; v < n; ++v) {\n    deg[v] = lc::row_degree(rp[v], rp[v + 1]);\n'
                   '    bin[v] = lc::bin_of(max_deg, deg[v]);\n  }\n}\n')
    so = d / "shim.so"
    cuda = os.path.join(os.path.dirname(os.path.dirname(_build.NVCC)), "include")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", _build.CSRC, "-I", cuda, str(src), "-o", str(so)])
    fn = ctypes.CDLL(str(so)).bins
    fn.argtypes = [ctypes.c_void_p, ctypes.c_int64] + [ctypes.c_void_p] * 3
    fn.restype = None

    def call(rp):
        n = rp.size - 1
        deg, b = np.zeros(n, np.int32), np.zeros(n, np.int32)
        fn(rp.ctypes.data, n, MAX_DEG.ctypes.data, deg.ctypes.data, b.ctypes.data)
        return deg, b

    return call


@pytest.mark.parametrize("name", list(row_pointers()))
def test_degree_is_the_difference_within_its_range(name, bins):
    rp = np.ascontiguousarray(row_pointers()[name], np.int64)
    deg, b = bins(rp)
    want = [min(max(int(y) - int(x), 0), (1 << 31) - 1) for x, y in zip(rp[:-1], rp[1:])]
    assert deg.tolist() == want
    assert np.array_equal(b, np.searchsorted(MAX_DEG, np.array(want, np.int64), side="left"))


def test_both_phases_take_the_degree_from_the_rule():
    """Counting and placing bin the one 32-bit degree (the counting phase's
    functor is held to that type; the records store it)."""
    src = open(os.path.join(_build.CSRC, "lc_bins.cu")).read()
    count = src[src.index("bins_count<kT>("):]
    assert "row_degree(" in count[:count.index(";")]
    for name in ("lc_bins.cu", "lc_level.cu"):
        src = open(os.path.join(_build.CSRC, name)).read()
        place = src[src.index("bins_place<kT>("):]
        assert "r.deg = row_degree(" in place[:place.index("});")], name


@pytest.mark.gpu
@pytest.mark.parametrize("name", [k for k in row_pointers() if k != "sound"])
def test_wild_row_ptr_is_refused_with_its_row(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2608_01503_gb300 as lc

    rp = np.ascontiguousarray(row_pointers()[name], np.int64).copy()
    n, nnz = rp.size - 1, 600
    rp[-1] = nnz
    beg, end = rp[:-1], rp[1:]
    first = int(np.argmax((end < beg) | (beg < 0) | (end > nnz)))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    rng = np.random.default_rng(4)
    args = (t(rp), t(rng.integers(0, n, nnz).astype(np.int32)), t(np.ones(nnz, np.int32)), t(np.ones(n, np.int64)))
    lab = torch.zeros(n, dtype=torch.int32, device="cuda")
    calls = [lambda: lc.lc_cluster(*args, 1, 50), lambda: lc.lc_cluster_leiden(*args, 1, 50),
             lambda: lc.lc_local_move(*args, 1, 50, lab), lambda: lc.lc_contract(*args, lab, 1),
             lambda: lc.lc_objective(*args, 1, 50, lab),
             lambda: lc.lc_cluster_batch(*args, np.array([0, n // 2, n]), [1, 1], [50, 50])]
    for k, call in enumerate(calls):
        with pytest.raises(lc.LCError) as e:
            call()
        assert e.value.code == 1, k
        if k not in (3, 5):  # lc_contract reports no row, a batch's edges may name an earlier one
            assert e.value.detail == first, k
    torch.cuda.synchronize()
