"""The symmetry check's two fingerprints are two checks: entries that agree in
one of them do not agree in the other for that reason."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2608_01503_gb300 import _build

M64 = (1 << 64) - 1
PHI = 0x9E3779B97F4A7C15


@pytest.fixture(scope="module")
def prints(tmp_path_factory):
    """edge_print of the library's own header, compiled for the host."""
    d = tmp_path_factory.mktemp("edge_print")
    src = d / "shim.cpp"
    src.write_text('#include "lc_edge_print.cuh"\n'
                   'extern "C" void prints(uint32_t lo, uint32_t hi, uint32_t w, unsigned long long *out) {\n'
                   '  const lc::EdgePrint p = lc::edge_print(lo, hi, w);\n  out[0] = p.a;\n  out[1] = p.b;\n}\n')
    so = d / "shim.so"
    cuda = os.path.join(os.path.dirname(os.path.dirname(_build.NVCC)), "include")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", _build.CSRC, "-I", cuda, str(src), "-o", str(so)])
    fn = ctypes.CDLL(str(so)).prints
    fn.argtypes = [ctypes.c_uint32] * 3 + [ctypes.c_void_p]
    fn.restype = None

    def call(lo, hi, w):
        out = (ctypes.c_uint64 * 2)()
        fn(lo, hi, w, out)
        return out[0], out[1]

    return call


def mix64(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return z ^ (z >> 31)


def unshift(z, s):
    """The x with x ^ (x >> s) == z."""
    x = z
    for _ in range(64 // s):
        x = z ^ (x >> s)
    return x


def unmix64(z):
    z = (unshift(z, 31) * pow(0x94D049BB133111EB, -1, 1 << 64)) & M64
    z = (unshift(z, 27) * pow(0xBF58476D1CE4E5B9, -1, 1 << 64)) & M64
    return unshift(z, 30)


def test_entries_that_agree_in_one_fingerprint_differ_in_the_other(prints):
    rng = np.random.default_rng(1)
    # two edges whose keys agree once the weights are mixed into them
    p, q = prints(70667, 14944714, 3), prints(1618112, 4160460, 5781)
    assert p[0] != q[0] and p[1] != q[1]
    # pairs made to agree in the first, and in the second
    for _ in range(2000):
        lo, hi = (int(x) for x in rng.integers(0, 1 << 31, 2))
        w, v = (int(x) for x in rng.integers(1, 1 << 31, 2))
        if v == w:
            continue
        m = mix64((lo << 32) | hi)
        key = unmix64(m ^ (w * PHI & M64) ^ (v * PHI & M64))
        p, q = prints(lo, hi, w), prints(key >> 32, key & 0xFFFFFFFF, v)
        assert p[0] == q[0] and p[1] != q[1]
        key = unmix64(m * (2 * w + 1) * pow(2 * v + 1, -1, 1 << 64) & M64)
        p, q = prints(lo, hi, w), prints(key >> 32, key & 0xFFFFFFFF, v)
        assert p[1] == q[1] and p[0] != q[0]


def test_unequal_weights_of_one_edge_differ(prints):
    rng = np.random.default_rng(2)
    for _ in range(300):
        lo, hi, w = (int(x) for x in rng.integers(1, 1 << 31, 3))
        a, b = prints(lo, hi, w)
        for bit in range(31):
            c, d = prints(lo, hi, w ^ (1 << bit))
            assert a != c and b != d


@pytest.mark.gpu
def test_entries_with_one_mixed_key_are_not_symmetric():
    """A graph of two entries, one stored from its lower end, one from its
    upper end, whose weight-mixed keys agree."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2608_01503_gb300 as lc

    n = 14944715
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[70667 + 1:] += 1    # 70667 -> 14944714, weight 3
    row_ptr[4160460 + 1:] += 1  # 4160460 -> 1618112, weight 5781
    col = torch.tensor([14944714, 1618112], dtype=torch.int32, device="cuda")
    ew = torch.tensor([3, 5781], dtype=torch.int32, device="cuda")
    with pytest.raises(lc.LCError) as e:
        lc.lc_objective(row_ptr, col, ew, torch.ones(n, dtype=torch.int64, device="cuda"), 1, 50,
                        torch.zeros(n, dtype=torch.int32, device="cuda"))
    assert e.value.code == 2
