"""Accuracy of the dense eigensolver where the way it computes shows: small matrices, rows of very
different size, close eigenvalues, the reduction in place, several reductions at once."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def fs():
    from paper_1907_06821_gb300 import build as b
    b.build()
    import paper_1907_06821_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(fs):
    with fs.Context((10.0, 10.0, 10.0), (16, 16, 16), 3.0, (0, 0, 0), np.zeros((16, 16, 16))) as c:
        yield c


def _herm(rng, n):
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return (a + a.conj().T) / (2 * np.sqrt(n))


@pytest.mark.parametrize("n", [2, 3, 4, 8])
def test_small_eigenvectors(ctx, n):
    """max |A z - w z| over a matrix's pairs, averaged over 60 matrices of norm 2 or less: below
    4 u ||A||.  (A backward-stable method stays within a few u ||A|| for a handful of rows; a
    perturbation of 10 eps ||T|| in one pivot of the inverse iteration gives 1.0 to 1.4e-15.)"""
    res = []
    for seed in range(60):
        A = _herm(np.random.default_rng(1000 * n + seed), n)
        w, Z = ctx.dense_eigh(A, m=n)
        Zl = Z.astype(np.clongdouble)
        res.append(float(np.abs(A.astype(np.clongdouble) @ Zl - Zl * w.astype(np.longdouble)).max()))
    assert np.mean(res) < 4 * U * 2.0


def test_multiples_of_the_unit_matrix(ctx):
    """T - w I has zero pivots throughout: the vectors are orthonormal and the values exact."""
    for n in (1, 2, 5, 40):
        w, Z = ctx.dense_eigh(3.0 * np.eye(n, dtype=complex), m=n)
        assert np.abs(w - 3.0).max() < 8 * U * 3.0
        assert np.abs(Z.conj().T @ Z - np.eye(n)).max() < 64 * n * U


# the triangular solves' products go to the tensor cores, and the matrices are scaled, from n = 315
# on; D runs up, down or mixed over six (1e-6 .. 1) or twelve decades (1e-6 .. 1e6)
@pytest.mark.parametrize("n,lo,hi", [(120, -6, 6), (314, -6, 6), (315, -6, 6), (600, -6, 6), (816, -6, 0)])
@pytest.mark.parametrize("order", ["up", "down", "mixed"])
def test_graded_b(ctx, n, lo, hi, order):
    """A = D A' D, B = D B' D: the eigenvalues are those of (A', B') and Y = D Z is B'-orthonormal.
    Cholesky and triangular substitution are indifferent to D, so the tolerance is that of the
    evenly scaled problem, 64 n u, of which the measured values are a few tenths of a percent: a
    hundredth of it, 0.64 n u, is asked for."""
    rng = np.random.default_rng(n)
    m = n // 3
    A, B = _herm(rng, n), np.eye(n) + 0.3 * _herm(rng, n)
    D = 10.0 ** np.linspace(lo, hi, n)
    D = {"up": D, "down": D[::-1], "mixed": rng.permutation(D)}[order]
    Ad, Bd = D[:, None] * A * D, D[:, None] * B * D
    A = ((Ad + Ad.conj().T) / 2) / D[:, None] / D
    B = ((Bd + Bd.conj().T) / 2) / D[:, None] / D
    w, Z = ctx.dense_eigh((Ad + Ad.conj().T) / 2, m=m, B=(Bd + Bd.conj().T) / 2)
    Y = D[:, None] * Z
    tol = 0.64 * n * U
    assert np.abs(Y.conj().T @ B @ Y - np.eye(m)).max() < tol
    assert np.abs(A @ Y - B @ Y * w).max() < tol


def test_scaled_and_indefinite_b(ctx):
    """B of any size by an exact power of two gives the same vectors; a B that is not positive
    definite is reported by its column, also with zeros and negative numbers on the diagonal."""
    from paper_1907_06821_gb300 import FSError, FS_ERR_NUMERIC
    rng = np.random.default_rng(5)
    A, B = _herm(rng, 48), np.eye(48) + 0.3 * _herm(rng, 48)
    w, Z = ctx.dense_eigh(A, m=48, B=B)
    w2, Z2 = ctx.dense_eigh(A, m=48, B=B * 2.0 ** -200)
    assert np.array_equal(w * 2.0 ** 200, w2) and np.array_equal(Z * 2.0 ** 100, Z2)
    for v in (0.0, -1.0, np.nan):
        C = B.copy()
        C[20, 20] = v
        with pytest.raises(FSError, match="column") as ei:
            ctx.dense_eigh(A, m=4, B=C)
        assert ei.value.code == FS_ERR_NUMERIC


# the reduction keeps its columns in shared memory up to 1,296 rows on 152 SMs, else in place;
# 2,048 is the largest size
@pytest.mark.parametrize("n", [1296, 1297, 2048])
def test_reduction_in_place(ctx, n):
    A = _herm(np.random.default_rng(n), n)
    w, Z = ctx.dense_eigh(A, m=7)
    tol = 64 * n * U
    assert np.abs(A @ Z - Z * w).max() < tol
    assert np.abs(Z.conj().T @ Z - np.eye(7)).max() < tol


# vectors of eigenvalues closer than 1e-13 of the norm are orthogonalised to one another in the
# inverse iteration, the others by the Cholesky QR pass
@pytest.mark.parametrize("gap", [1e-15, 5e-14, 2e-13, 1e-12, 1e-11, 1e-10])
def test_close_eigenvalues(ctx, gap):
    n, rng = 96, np.random.default_rng(17)
    Q = np.linalg.qr(_herm(rng, n))[0]
    lam = np.repeat(np.linspace(-1.0, 1.0, 12), 8) + gap * np.tile(np.arange(8), 12)
    A = (Q * lam) @ Q.conj().T
    A = (A + A.conj().T) / 2
    w, Z = ctx.dense_eigh(A, m=n)
    tol = 64 * n * U
    assert np.abs(w - np.linalg.eigvalsh(A)).max() < tol
    assert np.abs(A @ Z - Z * w).max() < tol
    assert np.abs(Z.conj().T @ Z - np.eye(n)).max() < tol


def test_several_reductions_at_once(fs):
    """Three threads, each with a context and eigenproblems whose reduction takes more than half of
    every SM's shared memory, so that two of them cannot be resident together: each runs to its end
    (a cooperative launch starts when all of its blocks fit) and none gives up waiting."""
    n, err = 1000, []
    mats = [_herm(np.random.default_rng(s), n) for s in range(3)]
    ref = [np.linalg.eigvalsh(A)[:8] for A in mats]

    def work(i):
        try:
            with fs.Context((10.0, 10.0, 10.0), (16, 16, 16), 3.0, (0, 0, 0), np.zeros((16, 16, 16))) as c:
                for _ in range(6):
                    w, _ = c.dense_eigh(mats[i], m=8)
                    assert np.abs(w - ref[i]).max() < 64 * n * U
        except BaseException as e:  # noqa: BLE001 - reported by the main thread
            err.append(e)
    th = [threading.Thread(target=work, args=(i,)) for i in range(3)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not err, err
