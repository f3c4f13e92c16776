"""The pivots' reciprocal square root against exact arithmetic and against the library's, over every exponent.

y' = y + y e (1/2 + 3/8 e), e = 1 - d y^2, with y the hardware's approximation of relative error at most 2^-19, so
|e| <= 2^-18.  In u = 2^-53: d y is rounded, which puts at most u into e and u / 2 into y'; the last fused multiply-add rounds
once more, u; the series' remainder is 5/16 |e|^3 < 0.2 u; products with e round far below.  Hence |error| <= 1.7 u, asserted
as 2 u.  The library's rsqrt is within one ulp, so the two are within three of each other.  Outside the biased exponents
100 .. 1900 the function is the library's, bit for bit (subnormals and infinity among them)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2006_06537_gb300 import build  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def kat(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("rsqrt") / "kat.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.SRC, "-shared", "-o", so,
                    os.path.join(HERE, "rsqrt_kat.cu")], check=True)
    lib = C.CDLL(so)

    def run(x):
        out = np.empty((2, len(x)))
        assert lib.rsqrt_kat(*(a.ctypes.data_as(C.c_void_p) for a in (x, out[0], out[1])), C.c_int(len(x))) == 0
        return out

    return run


def _doubles(exponents, per, seed):
    """`per` values of every biased exponent: the ends of its range and random mantissas."""
    m = np.random.default_rng(seed).integers(0, 1 << 52, (len(exponents), per), dtype=np.uint64)
    m[:, 0], m[:, 1], m[:, 2] = 0, (1 << 52) - 1, 1
    return ((np.asarray(exponents, np.uint64)[:, None] << np.uint64(52)) | m).ravel().view(np.float64)


def test_within_the_error_bound(kat):
    x = _doubles(np.arange(100, 1901), 40, 1)
    mine, lib = kat(x)
    worst = 0.0
    for d, y in zip(x.tolist(), mine.tolist()):
        md, ed = np.frexp(d)
        my, ey = np.frexp(y)
        num, s = int(md * 2.0 ** 53) * int(my * 2.0 ** 53) ** 2, 159 - int(ed) - 2 * int(ey)  # d y^2 = num / 2^s
        worst = max(worst, abs(num - (1 << s)) / (1 << (s + 1)))  # (d y^2 - 1) / 2
    assert worst <= 2 * 2.0 ** -53
    assert np.max(np.abs(mine.view(np.int64) - lib.view(np.int64))) <= 3


def test_the_library_beyond_the_range(kat):
    x = np.concatenate([_doubles(np.r_[0:100, 1901:2047], 40, 2), [np.inf, 5e-324, np.finfo(float).tiny, np.finfo(float).max]])
    x = x[x > 0]
    mine, lib = kat(x)
    assert np.array_equal(mine.view(np.int64), lib.view(np.int64))
