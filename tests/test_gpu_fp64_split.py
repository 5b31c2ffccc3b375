"""FP64 GEMMs on the tensor cores by error-free digit splitting (csrc/fs_oz.cu), through
the FP64 H application, whose nonlocal term takes that path from a few bands on.

Tolerance: both the library and the oracle sum up to npw products per projection in
FP64; with u = 2^-53 each is within about u sqrt(npw) of the exact sum relative to the
largest term, the FFTs within 8 u log2(N): 4 (sqrt(npw) + 8 log2 N) u covers both sides.
"""
import numpy as np
import pytest

import fs_inputs as fi
from gpu_helpers import rel_err
from oracle import planewave as pw

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fs():
    from paper_1907_06821_gb300 import build as b
    b.build()
    import paper_1907_06821_gb300 as m
    return m


def _psi(nb, npw, seed=5):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((nb, npw)) + 1j * rng.standard_normal((nb, npw))


# tiles: 128 rows x 32 columns x chains of 64 k; 33 atoms x 4 = 132 projectors (one tile and
# four rows), bands at the edges of the column tiles
@pytest.mark.parametrize("nb", [12, 31, 32, 33, 65, 130])
@pytest.mark.parametrize("natom,widths", [(33, (1.0,)), (13, (0.8, 1.2))])
def test_apply_matches_oracle(fs, nb, natom, widths):
    w = fi.make_box(L=(13.0, 13.0, 17.0), n=(24, 24, 32), ecut=6.0, k=(0.02, -0.01, 0.03), natom=natom,
                    widths=widths, lattice=4.0, nstates=4, e_ref=0.2, seed=21)
    with fs.Context.from_workload(w) as c:
        psi = _psi(nb, c.npw)
        out = c.apply_H(torch.as_tensor(psi, device="cuda"), shift=0.1).cpu().numpy()
        ref = pw.Hamiltonian(w).apply(psi) - 0.1 * psi
        tol = 4 * (np.sqrt(c.npw) + 8 * np.log2(24 * 24 * 32)) * 2.0 ** -53
        assert rel_err(out, ref) < tol


def test_scales_and_non_finite_rows(fs):
    w = fi.make_box(L=(13.0, 13.0, 17.0), n=(24, 24, 32), ecut=6.0, natom=33, widths=(1.0,), lattice=4.0,
                    nstates=4, e_ref=0.2, seed=22)
    with fs.Context.from_workload(w) as c:
        psi = _psi(16, c.npw)
        a = c.apply_H(torch.as_tensor(psi, device="cuda")).cpu().numpy()
        f = 2.0 ** np.linspace(-400, 400, 16).astype(int)
        b = c.apply_H(torch.as_tensor(psi * f[:, None], device="cuda")).cpu().numpy()
        assert np.array_equal(b, a * f[:, None])      # powers of two pass through exactly
        psi[3, 17] = np.nan
        psi[5, 100] = np.inf
        psi[7] = 0.0
        with np.errstate(invalid="ignore"):
            d = c.apply_H(torch.as_tensor(psi, device="cuda")).cpu().numpy()
        keep = [i for i in range(16) if i not in (3, 5, 7)]
        assert np.array_equal(d[keep], a[keep])
        assert not np.isfinite(d[3]).any() and not np.isfinite(d[5]).any() and not d[7].any()


def test_row_maxima_at_the_top_of_the_digit_range(fs):
    # the largest component of a row around 127.5 / 128 of a power of two, where seven signed
    # digits end (0x7F7F7F7F7F7F7F = 0.996078 2^55) and the next exponent is taken
    w = fi.make_box(L=(13.0, 13.0, 17.0), n=(24, 24, 32), ecut=6.0, natom=33, widths=(1.0,), lattice=4.0,
                    nstates=4, e_ref=0.2, seed=23)
    top = [0.992, 0.9921875, 0.99606, 0.996078, 0.9960784, 0.996080, 0.99609, 0.99609375, 0.9961, 1 - 2.0 ** -53,
           -0.99608, -(1 - 2.0 ** -53)]
    with fs.Context.from_workload(w) as c:
        psi = _psi(len(top), c.npw)
        psi /= np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=1)[:, None] * 1.1
        for i, t in enumerate(top):
            psi[i, 11 * i] = t + 0.25j if i % 2 else 0.25 + 1j * t
        out = c.apply_H(torch.as_tensor(psi, device="cuda")).cpu().numpy()
        ref = pw.Hamiltonian(w).apply(psi)
        tol = 4 * (np.sqrt(c.npw) + 8 * np.log2(24 * 24 * 32)) * 2.0 ** -53
        for i in range(len(top)):
            assert rel_err(out[i], ref[i]) < tol, top[i]
