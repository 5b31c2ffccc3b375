"""Accuracy of the dense eigensolver where the way it computes shows: small matrices."""
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
