"""Host tables of the FP64 pair kinematics, compiled for the host alone: every entry of the azimuth and logarithm tables is its
value rounded once (half an ulp, and a thousandth for the reference's own rounding in the host's long double)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N97, TURN, LN = 9 * 64, 256, 128
HALF_ULP = 0.5 + 1e-3


@pytest.fixture(scope="module")
def tables(tmp_path_factory):
    d = tmp_path_factory.mktemp("tables")
    src = d / "t.cpp"
    src.write_text('#include "mcc_tables.h"\nextern "C" void f64(double* o) { mcc::f64_tables(o); }\n'
                   'extern "C" int sizes(int* o) { o[0] = mcc::kF64N97; o[1] = mcc::kF64Turn; o[2] = mcc::kF64Ln;\n'
                   'return (int)mcc::kF64TabDoubles; }\n')
    so = d / "t.so"
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2407_19151_gb300", "csrc"), "-o", str(so), str(src)], check=True)
    L = ctypes.CDLL(str(so))
    sizes = (ctypes.c_int * 3)()
    n = L.sizes(sizes)
    assert list(sizes) == [N97, TURN, LN] and n == 24 * N97 + 2 * TURN + 2 * LN
    out = np.zeros(n)
    L.f64(out.ctypes.data_as(ctypes.c_void_p))
    return out


def _ulps(got, want):
    """Distance in units of the last place of `got` (long double arithmetic)."""
    assert np.finfo(np.longdouble).nmant >= 60
    return np.abs(got.astype(np.longdouble) - want) / np.spacing(np.maximum(np.abs(got), 1e-300)).astype(np.longdouble)


def _turn(i):
    """cos of i/256 turn in long double, the angle reduced to an eighth of a turn in whole numbers."""
    i = abs((i + 128) % 256 - 128)
    sign = 1 if i <= 64 else -1
    i = min(i, 128 - i)
    pi = 4 * np.arctan(np.longdouble(1))
    return sign * (np.cos(pi * i / 128) if i <= 32 else np.sin(pi * (64 - i) / 128))


def test_turn_entries(tables):
    turn = tables[24 * N97:24 * N97 + 2 * TURN].reshape(-1, 2)
    want = np.array([[_turn(i), _turn(i - 64)] for i in range(TURN)], dtype=np.longdouble)
    zero = want == 0
    assert zero.sum() == 4 and (turn[zero] == 0).all()
    assert _ulps(turn[~zero], want[~zero]).max() <= HALF_ULP


def test_logarithm_entries(tables):
    r, l = tables[24 * N97 + 2 * TURN:].reshape(-1, 2).T
    one = r == 1.0
    assert one.sum() == 2 and (l[one] == 0).all()
    assert _ulps(l[~one], -np.log(r[~one].astype(np.longdouble))).max() <= HALF_ULP
