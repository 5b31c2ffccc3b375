"""Sizes at the edges of the tiles and dispatch rules of the dense algebra, the FP32-stage
products and the training step.

Tolerances: eigenpairs and orthogonality to 64 n u (u = 2^-53; backward-stable methods stay
within a small multiple of n u ||A||, ||A|| about 2 here); FP32-stage products keep about
22 bits per product and FP32 sums, 8 sqrt(K) 2^-24 relative to the largest value; gradient
sums keep FP32 products, 64 * 2^-24 of the largest entry.
"""
import numpy as np
import pytest

import fs_inputs as fi
from gpu_helpers import rel_err
from oracle import mlp
from oracle import planewave as pw

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fs():
    from paper_1907_06821_gb300 import build as b
    b.build()
    import paper_1907_06821_gb300 as m
    return m


def _ctx(fs):
    return fs.Context((10.0, 10.0, 10.0), (16, 16, 16), 3.0, (0, 0, 0), np.zeros((16, 16, 16)))


def _herm(rng, n):
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return (a + a.conj().T) / (2 * np.sqrt(n))


# panels and diagonal blocks of 128 (32 within them), row chunks of 128 / 256 / 512 / 1024 in the
# reduction, columns in shared memory up to 1,216
@pytest.mark.parametrize("n,m", [(1, 1), (2, 1), (33, 33), (127, 127), (128, 40), (129, 129), (256, 9), (257, 200),
                                 (513, 30), (1025, 17), (1217, 5)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 300, 2.0 ** -300])
def test_dense_eigh_edges(fs, n, m, scale):
    if scale != 1.0 and n > 300:
        pytest.skip("scales on the smaller sizes")
    rng = np.random.default_rng(n)
    A, B = _herm(rng, n), np.eye(n) + 0.3 * _herm(rng, n)
    tol = 64 * n * 2.0 ** -53
    with _ctx(fs) as c:
        w, Z = c.dense_eigh(A * scale, m=m)
        assert np.abs(w / scale - np.linalg.eigvalsh(A)[:m]).max() < tol
        assert np.abs(A @ Z - Z * (w / scale)).max() < tol
        assert np.abs(Z.conj().T @ Z - np.eye(m)).max() < tol
        w, Z = c.dense_eigh(A, m=m, B=B)
        assert np.abs(A @ Z - B @ Z * w).max() < tol
        assert np.abs(Z.conj().T @ B @ Z - np.eye(m)).max() < tol


# 64 and 128 columns a tile, 128 rows a tile; projector sets of 1, 4 and 5 per atom (phases are
# shared by fours), stored and generated
@pytest.mark.parametrize("nb", [1, 8, 127, 129, 257])
@pytest.mark.parametrize("nproj", [1, 4, 5])
def test_fp32_products_edges(fs, nb, nproj):
    w = fi.make_box(L=(11.0, 12.0, 13.0), n=(20, 24, 24), ecut=5.0, k=(0.01, 0.02, -0.03), natom=33, widths=(1.0,),
                    lattice=3.5, nstates=4, e_ref=0.2, seed=31)
    w.proj = (list(w.proj) + [(0, 0, 0.8)])[:nproj] if nproj != 4 else w.proj
    rng = np.random.default_rng(1)
    D = rng.uniform(0.1, 0.5, (33, nproj, nproj))
    w.D = (D + D.transpose(0, 2, 1)) / 2
    H = pw.Hamiltonian(w)
    out = {}
    for mode in (fs.FS_PROJ_STORED, fs.FS_PROJ_GENERATED):
        with fs.Context.from_workload(w, precision=fs.FS_MIXED, projectors=mode) as c:
            x = (rng.standard_normal((nb, c.npw)) + 1j * rng.standard_normal((nb, c.npw))).astype(np.complex64)
            # rows of very different size keep their relative accuracy
            x *= (10.0 ** rng.uniform(-12, 12, nb)).astype(np.float32)[:, None]
            y = c.apply_H(torch.as_tensor(x, device="cuda")).cpu().numpy()
            ref = H.apply(x.astype(np.complex128))
            out[mode] = max(rel_err(y[i], ref[i]) for i in range(nb))
    assert max(out.values()) < 8 * np.sqrt(ref.shape[1]) * 2.0 ** -24


# tiles of 64 rows, one block per SM (152 x 64 rows in one round)
@pytest.mark.parametrize("rows", [1, 31, 63, 64, 65, 9728, 9729])
def test_gradient_row_edges(fs, rows):
    rng = np.random.default_rng(rows)
    theta = mlp.init_params(3)
    theta[-129:] = rng.uniform(-0.1, 0.1, 129)
    F = rng.normal(0, 0.5, (rows, 4)).astype(np.float32)
    zt, wt = rng.normal(0, 0.5, rows).astype(np.float32), rng.uniform(0.1, 1, rows).astype(np.float32)
    with _ctx(fs) as c:
        c.precond_weights(theta.astype(np.float32))
        loss, g = c.precond_loss_grad(*[torch.as_tensor(v, device="cuda") for v in (F, zt, wt)])
    th = theta.astype(np.float32).astype(np.float64)
    ref = _loss_grad(th, F.astype(np.float64), zt.astype(np.float64), wt.astype(np.float64))
    assert abs(loss - ref[0]) < 64 * 2.0 ** -24 * ref[0]
    assert rel_err(g.cpu().numpy().astype(np.float64), ref[1]) < 64 * 2.0 ** -24


def _loss_grad(theta, F, zt, wt):
    """Forward with BF16-rounded weights, backward with the master weights, FP64."""
    layers = mlp.unpack(theta)
    h = [F]
    for i, (W, b) in enumerate(layers):
        p = h[-1] @ mlp.bf16_round(W).T + b
        h.append(np.tanh(p) if i < 3 else p)
    r = h[4][:, 0] - zt
    g, grads = (2 * wt * r / wt.sum())[:, None], []
    for i in (3, 2, 1, 0):
        grads.append(np.concatenate([(g.T @ h[i]).ravel(), g.sum(0)]))
        if i:
            g = (g @ layers[i][0]) * (1 - h[i] ** 2)
    return (wt * r * r).sum() / wt.sum(), np.concatenate(grads[::-1])
