"""The fit's products one by one against 64-bit-mantissa sums: no further off than the FP64 kernel on operands of every
kind, and exact where they are exact."""
import glob
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2511_20687_gb300")


@pytest.fixture(scope="module")
def product(tmp_path_factory):
    from paper_2511_20687_gb300 import build_lib
    build_lib.build(force=not os.path.isdir(build_lib.BUILD))
    d = tmp_path_factory.mktemp("products")
    exe = str(d / "check")
    subprocess.run([build_lib.nvcc(), *build_lib.ARCH, "-O2", "-std=c++17", "-I", build_lib.INCLUDE, "-I", build_lib.CSRC,
                    "-o", exe, os.path.join(ROOT, "tests/split_product_check.cu"),
                    *sorted(glob.glob(os.path.join(build_lib.BUILD, "*.o")))], check=True)

    def run(A, B, layout):
        m, k = A.shape
        n = B.shape[0]
        with open(d / "in", "wb") as f:
            np.array([m, n, k, layout], np.int32).tofile(f)
            np.ascontiguousarray(A).tofile(f)
            np.ascontiguousarray(B).tofile(f)
        subprocess.run([exe, str(d / "in"), str(d / "out")], check=True)
        return np.fromfile(d / "out").reshape(2, m, n)

    return run


def operands(kind, m, n, k, rng):
    A, B = rng.standard_normal((m, k)), rng.standard_normal((n, k))
    if kind.startswith("rows"):        # every third column of A dominates, by 1e3 or 1e6, and is missing in most of B
        A[:, ::3] *= float(kind[4:])
        B[::2, ::3] *= 1e-9
    elif kind == "decay":              # magnitudes over many decades along k
        A *= 10.0 ** (-12 * np.arange(k) / k)
        B *= 10.0 ** (-12 * np.arange(k)[::-1] / k)
    elif kind == "outlier":            # a few large elements in otherwise even rows
        A[:, k // 2] *= 1e5
    elif kind == "apart":              # operands that hardly overlap
        A[:, : k // 2] *= 1e-10
        B[:, k // 2:] *= 1e-10
    elif kind == "positive":
        A, B = np.abs(A), np.abs(B)
    elif kind == "scales":             # every row its own power of ten
        A *= 10.0 ** rng.integers(-60, 60, (m, 1))
        B *= 10.0 ** rng.integers(-60, 60, (n, 1))
    return A, B


KINDS = ["random", "rows1e3", "rows1e6", "decay", "outlier", "apart", "positive", "scales"]
SIZES = [(512, 512, 16), (512, 512, 64), (300, 200, 127), (300, 200, 128), (260, 65, 300), (70, 70, 1025), (64, 64, 4100),
         (3, 130, 20011)]


def exact(A, B):
    return A.astype(np.longdouble) @ B.T.astype(np.longdouble)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("m,n,k", SIZES)
def test_no_further_off_than_fp64(product, kind, m, n, k):
    """Root mean square over the entries of the error relative to |A||B|, by row of A: no row is further off than
    the FP64 kernel by more than the scatter of a row's n entries allows (2, and a half of a rounding of the result)."""
    rng = np.random.default_rng(21)
    A, B = operands(kind, m, n, k, rng)
    layout = SIZES.index((m, n, k)) % 3
    C, F = product(A, B, layout)
    X, S = exact(A, B), np.abs(A) @ np.abs(B).T
    e, f = (np.sqrt(np.mean(np.asarray((Y - X) / S, float) ** 2, axis=1)) for Y in (C, F))
    assert np.sqrt(np.mean(e ** 2)) <= np.sqrt(np.mean(f ** 2)) * 1.02
    assert (e <= 2 * f + 2.0 ** -55).all()


def value(digits):
    return sum(d << (8 * (6 - i)) for i, d in enumerate(digits))


def kept(a, b):
    """The digit products of weight 7 and below, in units of 2^-108."""
    return sum(x * y << (8 * (12 - i - j)) for i, x in enumerate(a) for j, y in enumerate(b) if i + j <= 7)


@pytest.mark.gpu
@pytest.mark.parametrize("place", [1, 2, 3, 4])
def test_largest_digit_sums(product, place):
    """Digits of 127 throughout (the last one even, for 53 bits): over 128 of k the seven products of the last weight sum
    to 0.86 of 2^24, by odd steps, so an accumulator that is emptied too late loses units.  The second half of the
    chunk subtracts almost the same, which leaves a result of few bits: it is compared with the whole-number sum of the
    kept products.  Only the accumulator of weights 6 and 7 rounds, below one unit (2^48) in each of its 13 x 64 steps;
    a unit of weight 5 is 256 of them."""
    a = [33, 127, 127, 127, 127, 127, 126]
    b = list(a)
    b[place] -= 1
    m, n, k = 64, 128, 1024
    A = np.full((m, k), value(a) * 2.0 ** -54)
    B = np.full((n, k), value(a) * 2.0 ** -54)
    B[:, k // 2:] = -value(b) * 2.0 ** -54
    want = k // 2 * (kept(a, a) - kept(a, b))
    for sign in (1.0, -1.0):
        C, _ = product(A, sign * B, 0)
        assert len(np.unique(C)) == 1
        assert abs(int(sign * C[0, 0] * 2.0 ** 108) - want) <= 13 * 64 * 2 ** 48


@pytest.mark.gpu
@pytest.mark.parametrize("layout", [0, 1, 2, 3])
def test_whole_numbers_are_exact(product, layout):
    """Integers of up to 2^20 over 2000 of k: every sum is below 2^52 and exact in FP64, so it is here."""
    rng = np.random.default_rng(23)
    A = rng.integers(-2 ** 20, 2 ** 20, (100, 2000)).astype(float)
    B = A if layout == 3 else rng.integers(-2 ** 20, 2 ** 20, (90, 2000)).astype(float)
    C, _ = product(A, B, layout)
    assert np.array_equal(C, np.asarray(exact(A, B), float))


@pytest.mark.gpu
@pytest.mark.parametrize("layout", [0, 2, 3])
def test_special_values(product, layout):
    """Infinities, NaN, subnormals, zero rows and products out of the normal range: what the FP64 kernel gives."""
    rng = np.random.default_rng(25)
    A = rng.standard_normal((200, 1500))
    B = A if layout == 3 else rng.standard_normal((150, 1500))
    A[3, 5] = np.inf
    A[70, 1400] = np.nan
    A[130] = 0.0
    A[131] *= 1e-310
    A[132] *= 1e-160
    A[133] *= 1e160
    B[140] *= 1e-200
    C, F = product(A, B, layout)
    assert np.array_equal(np.isnan(C), np.isnan(F)) and np.array_equal(np.isinf(C), np.isinf(F))
    assert np.isinf(C[3]).sum() > 100 and np.isnan(C[70]).all()
    ok = np.isfinite(F)
    assert (C[130][ok[130]] == 0.0).all()
    rows = [131, 132, 133]
    assert np.array_equal(C[rows][ok[rows]], F[rows][ok[rows]])
