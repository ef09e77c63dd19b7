"""The short device functions that stand for longer ones, over their whole range where
that can be walked through (every FP32 number, every input word) and over random
numbers of every exponent where it cannot.

The FP32 and BF16 ones are the same bits everywhere; strip_recip within the range its
comment states (2^-126 .. 2^126).  The FP64 reciprocal and face are correct to about
2^-88 before the last rounding, so they miss the IEEE quotient once in some 2^34: of
2^30 numbers (2^28 of the widest range) at most three differ, none by more than an ulp.
"""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CASES = ["gelu", "normal", "widen", "narrow", "twice", "strip_recip", "recip", "diagonal", "face", "face_far"]


@pytest.fixture(scope="module")
def compare(tmp_path_factory):
    from paper_1910_04727_gb300 import build as B
    so = str(tmp_path_factory.mktemp("short") / "short.so")
    r = subprocess.run([B._nvcc()] + B.ARCH + B.FLAGS + ["-shared", os.path.join(HERE, "short_functions.cu"), "-o", so],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(so)

    def run(name, count):
        out = (ctypes.c_ulonglong * 2)()
        assert lib.compare(CASES.index(name), ctypes.c_uint64(count), out) == 0
        return out[0], out[1]
    return run


@pytest.mark.parametrize("name,log2", [("gelu", 32), ("normal", 23), ("widen", 32), ("narrow", 32), ("twice", 30),
                                       ("strip_recip", 32), ("recip", 32)])
def test_the_same_bits(compare, name, log2):
    assert compare(name, 1 << log2) == (0, 0)


@pytest.mark.parametrize("name,log2", [("diagonal", 30), ("face", 30), ("face_far", 28)])
def test_at_most_a_rounding_apart(compare, name, log2):
    differ, far = compare(name, 1 << log2)
    assert differ <= 3 and far == 0
