"""Single pieces of the library on the GPU, called directly (tests/native_pieces.cu): the symmetric
eigensolver on either side of its border (96 rows)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ENAN = -4


@pytest.fixture(scope="module")
def native(tmp_path_factory):
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    so = str(tmp_path_factory.mktemp("native") / "native_pieces.so")
    subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-shared", os.path.join(HERE, "native_pieces.cu"),
                    b.LIB, "-Xlinker", f"-rpath={os.path.dirname(b.LIB)}", "-o", so], check=True)
    return C.CDLL(so)


def _p(x):
    return x.ctypes.data_as(C.c_void_p)


def _eig(native, A, wmin=-1e300):
    """Status, all eigenvalues, the vectors of those at or above wmin."""
    A, m = np.ascontiguousarray(A), A.shape[0]
    w, V, nk = np.zeros(m), np.zeros(m * m), C.c_int()
    st = native.np_eig_above(_p(A), m, C.c_double(wmin), _p(w), _p(V), C.byref(nk))
    return st, w, V[:m * nk.value].reshape(m, nk.value)


def _spd(m, seed=0):
    A = np.random.default_rng(seed).standard_normal((m, m))
    return A @ A.T


@pytest.mark.parametrize("m,bad", [(m, b) for m in (2, 3, 8, 33, 96) for b in (np.nan, np.inf)] +
                         [(100, np.nan)])
def test_matrix_that_is_not_finite_is_an_error(native, m, bad):
    """Every place of the first row (the later rows receive it through the first reflector, unless
    the value sits right of the subdiagonal there) and the last diagonal element."""
    for i, j in {(0, 0), (0, 1), (0, min(2, m - 1)), (0, m - 1), (m - 1, m - 1)}:
        A = _spd(m)
        A[i, j] = A[j, i] = bad
        assert _eig(native, A)[0] == ENAN, (i, j)


EPS = 2.0 ** -52


@pytest.mark.parametrize("m", [1, 2, 8, 32, 96])
@pytest.mark.parametrize("scale", [1.0, 1e-3, 1e-6, 1e-12, 1e-100, 1e100])
def test_small_matrix_keeps_its_digits(native, m, scale):
    """Eigenvalues of up to 96 rows to the backward error of a Householder reduction (4 m eps, as
    much again for the reference) relative to the norm, whatever the norm is; vectors to 20 m eps."""
    A = _spd(m, m) * scale
    st, w, V = _eig(native, A)
    ref = np.linalg.eigvalsh(A)
    assert st == 0
    assert np.abs(w - ref).max() <= 8 * m * EPS * np.abs(ref).max()
    assert np.abs(V.T @ V - np.eye(m)).max() <= 20 * m * EPS
    assert np.abs(A @ V - V * w).max() <= 20 * m * EPS * np.abs(ref).max()


@pytest.mark.parametrize("m", [1, 7, 40, 96])
@pytest.mark.parametrize("power", [-200, -20, 20, 200])
def test_small_matrix_scaled_by_a_power_of_two(native, m, power):
    """Scaling by a power of two changes no digit: eigenvalues, kept vectors and their count at a
    cut that scales along."""
    A, f = _spd(m, 5 + m), 2.0 ** power
    cut = 0.3 * m
    a, b = _eig(native, A, cut), _eig(native, A * f, cut * f)
    assert a[0] == b[0] == 0
    assert np.array_equal(a[1] * f, b[1])
    assert np.array_equal(a[2], b[2])
