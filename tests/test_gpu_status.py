"""A device-side wait that gave up is reported by the call that ran into it, whatever the call
computes, and by no later one.

The library's bounded wait runs out on a barrier that nothing completes and leaves the error flag
raised (fs_wait_selftest_pending), as a wait inside the call would; the call must return
FS_ERR_TIMEOUT, also where its numbers then look singular or not positive definite, and the next
one must succeed.
"""
import numpy as np
import pytest

import fs_inputs as fi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fs():
    from paper_1907_06821_gb300 import build as b
    b.build()
    import paper_1907_06821_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(fs):
    w = fi.make_config("tiny")
    with fs.Context.from_workload(w, precision=fs.FS_MIXED) as c:
        c.workload = w
        yield c


def _cuda(x, dtype=np.complex128):
    t = torch.as_tensor(np.asarray(x, dtype=dtype), device="cuda")
    torch.cuda.synchronize()  # the library's stream does not wait for torch's
    return t


def _block(c, n, seed=3):
    return fi.raw_start_block(n, c.npw, seed)


def _features(c, dt):
    X = _cuda(np.linalg.qr(_block(c, 4).T)[0].T, dt)
    c.precond_features(c.workload.e_ref, _cuda(_block(c, 2), dt), np.array([0.1, 0.2]), X=X[:2].contiguous(), Xref=X)


def _kinterp(c):
    P = _cuda(np.linalg.qr(_block(c, 5).T)[0].T)
    c.kinterp(0.3, np.arange(4.0), P[:4].contiguous(), np.arange(5.0), P)


def _kinterp_deficient(c):
    P = np.linalg.qr(_block(c, 5).T)[0].T
    Q = P[:4].copy()
    Q[2] = 0.0
    c.kinterp(0.3, np.arange(4.0), _cuda(Q), np.arange(5.0), _cuda(P))


def _loss(c):
    one = _cuda(np.ones(70), np.float32)
    c.precond_loss_grad(_cuda(np.zeros((70, 4)), np.float32), one, one)


CALLS = {
    "spectral_bounds": lambda c: c.spectral_bounds(4),
    "precond_features_fp64": lambda c: _features(c, np.complex128),
    "precond_features_fp32": lambda c: _features(c, np.complex64),
    "precond_eval": lambda c: c.precond_eval(_cuda(np.zeros((70, 4)), np.float32)),
    "precond_loss_grad": _loss,
    "kinterp": _kinterp,
    "dense_eigh": lambda c: c.dense_eigh(np.eye(6, dtype=complex)),
    "apply_H_fp64": lambda c: c.apply_H(_cuda(_block(c, 3))),
    "apply_H_fp32": lambda c: c.apply_H(_cuda(_block(c, 3), np.complex64)),
    "chebfd": lambda c: c.chebfd(-0.5, 1.0, -8.0, 9.0, 8, 6, 1),
    "linear_solve": lambda c: c.linear_solve(_cuda(_block(c, 2)), 0.0, tol=1e-3, maxit=3, allow_unconverged=True),
    "solve": lambda c: c.solve(c.workload.e_ref, 4, tol=1e-4),
    "solve_lowest": lambda c: c.solve_lowest(4, tol=1e-3),
    "autotune": lambda c: c.autotune(),
}


@pytest.mark.parametrize("name", list(CALLS))
def test_pending_timeout_is_reported_once(fs, ctx, name):
    ctx.wait_selftest(512, pending=True)
    with pytest.raises(fs.FSError) as ei:
        CALLS[name](ctx)
    assert ei.value.code == fs.FS_ERR_TIMEOUT
    CALLS[name](ctx)


BAD = {
    "kinterp": _kinterp_deficient,
    "dense_eigh": lambda c: c.dense_eigh(np.eye(6, dtype=complex), B=-np.eye(6, dtype=complex)),
}


@pytest.mark.parametrize("name", list(BAD))
def test_timeout_before_a_numeric_error(fs, ctx, name):
    ctx.wait_selftest(512, pending=True)
    with pytest.raises(fs.FSError) as ei:
        BAD[name](ctx)
    assert ei.value.code == fs.FS_ERR_TIMEOUT
    with pytest.raises(fs.FSError) as ei:
        BAD[name](ctx)
    assert ei.value.code == fs.FS_ERR_NUMERIC
