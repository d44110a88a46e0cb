"""Single pieces of the library on the GPU, called directly (tests/native_pieces.cu): the symmetric
eigensolver on either side of its border (96 rows), and the reciprocal and the root that stand in
for a division and a square root."""
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


def _eig(native, A, wmin=-1e300, block=None):
    """Status, all eigenvalues, the vectors of those at or above wmin; up to 96 rows in the
    one-block solver unless said otherwise."""
    A, m = np.ascontiguousarray(A), A.shape[0]
    w, V, nk = np.zeros(m), np.zeros(m * m), C.c_int()
    st = native.np_eig_above(_p(A), m, C.c_double(wmin), _p(w), _p(V), C.byref(nk),
                             int(m <= 96 if block is None else block))
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


def _repeated(kind, m, rng):
    """Eigenvalues with many equal ones: a projector's null space, two values, three clusters of
    different sizes, and one beside a close pair."""
    if kind == "rank":
        w = np.concatenate([np.zeros(m - m * 3 // 5), rng.uniform(0.1, 4.0, m * 3 // 5)])
    elif kind == "two":
        w = np.where(np.arange(m) % 2, 1.0, -0.5)
    elif kind == "three":
        w = np.repeat([0.3, 0.7, 2.0], [m // 4, m // 4, m - 2 * (m // 4)])
    else:
        w = np.concatenate([np.full(m - 3, 1.0), [1.0 + 1e-6, 3.0, 3.5]])
    Q = np.linalg.qr(rng.standard_normal((m, m)))[0]
    A = (Q * w) @ Q.T
    return 0.5 * (A + A.T)


@pytest.mark.parametrize("m", [8, 16, 31, 32, 60, 80, 96])
@pytest.mark.parametrize("kind", ["rank", "two", "three", "close"])
def test_equal_eigenvalues(native, m, kind):
    """Residual and orthogonality to 20 m eps of the norm, where the vectors of equal eigenvalues
    come from independent starts; ten matrices each."""
    for seed in range(10):
        A = _repeated(kind, m, np.random.default_rng(seed))
        st, w, V = _eig(native, A)
        norm = np.abs(w).max()
        assert st == 0
        assert np.abs(V.T @ V - np.eye(m)).max() <= 20 * m * EPS
        assert np.abs(A @ V - V * w).max() <= 20 * m * EPS * norm, seed


@pytest.mark.parametrize("m", [97, 128, 200, 300])
@pytest.mark.parametrize("kind", ["rank", "two", "three", "close"])
def test_equal_eigenvalues_large(native, m, kind):
    """The same on the large path.  Of a unit start Gram-Schmidt leaves 1 / sqrt(k) in a space of k
    equal eigenvalues and may leave a tenth of 1 / k of the worst: m eps (the reduction) times 10 k,
    k up to 150, is 1e-10 of the norm; orthogonality is restored to 1e-13 afterwards."""
    for seed in range(5):
        A = _repeated(kind, m, np.random.default_rng(seed))
        st, w, V = _eig(native, A)
        assert st == 0
        assert np.abs(V.T @ V - np.eye(m)).max() <= 1e-12
        assert np.abs(A @ V - V * w).max() <= 1e-10 * np.abs(w).max(), seed


@pytest.mark.parametrize("m", [1, 5, 32, 96])
def test_diagonal_and_decoupled(native, m):
    """No coupling at all, equal elements among them, and two equal blocks."""
    rng = np.random.default_rng(m)
    d = np.round(rng.uniform(-2, 2, m), 1)
    st, w, V = _eig(native, np.diag(d))
    assert st == 0
    assert np.abs(w - np.sort(d)).max() <= 4 * EPS * np.abs(d).max()
    assert np.abs(np.diag(d) @ V - V * w).max() <= 20 * EPS * np.abs(d).max()
    if m % 2 == 0:
        A = np.kron(np.eye(2), _spd(m // 2, 1))
        st, w, V = _eig(native, A)
        assert st == 0
        assert np.abs(V.T @ V - np.eye(m)).max() <= 20 * m * EPS
        assert np.abs(A @ V - V * w).max() <= 20 * m * EPS * np.abs(w).max()


def _arguments():
    """Mantissas over [1, 4) with every edge, exponents over the range of a denominator or norm."""
    rng = np.random.default_rng(3)
    x = rng.uniform(1.0, 4.0, 1 << 20)
    x[:3] = 1.0, np.nextafter(2.0, 0.0), np.nextafter(4.0, 0.0)
    return np.concatenate([x * 2.0 ** e for e in (-300, -20, -1, 0, 1, 10, 300)])


def test_reciprocal(native):
    """0.5 units for the last rounding and 2^-60 relative (below 2^-7 units) for the series."""
    x = _arguments()
    x = np.concatenate([x, -x])
    y = np.zeros_like(x)
    assert native.np_recip(_p(x), C.c_long(x.size), _p(y)) == 0
    exact = 1 / x.astype(np.longdouble)
    assert float((np.abs(y - exact) / np.spacing(np.abs(y))).max()) <= 0.51


def test_root_and_reciprocal_root(native):
    """Relative to 2^-53: 1 for the last rounding, 1/2 for the product's, 2^-5 for the series."""
    x = _arguments()
    r, ir = np.zeros_like(x), np.zeros_like(x)
    assert native.np_root(_p(x), C.c_long(x.size), _p(r), _p(ir)) == 0
    exact = np.sqrt(x.astype(np.longdouble))
    for got, ref in ((r, exact), (ir, 1 / exact)):
        assert float((np.abs(got - ref) / ref).max()) <= 1.6 * 2.0 ** -53
