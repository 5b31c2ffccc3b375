"""Contexts made and destroyed in sequence, in number, and around a reset of the device.

The error flags of a process's contexts share pinned pages, one of which stays when the last context
goes: it must be there for the next one, and must not be used when the device was reset in between.
The reset runs in a process of its own, without torch (fs_dense_eigh and fs_solve take host buffers).
"""
import os
import subprocess
import sys
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import ctypes
import numpy as np
import fs_inputs as fi
import paper_1907_06821_gb300 as fs

def use():
    rng = np.random.default_rng(1)
    a = rng.standard_normal((600, 600)) + 1j * rng.standard_normal((600, 600))
    A = (a + a.conj().T) / 2
    B = np.eye(600) + 0.01 * A
    w = fi.make_config("tiny")
    with fs.Context.from_workload(w, precision=fs.FS_MIXED) as c:
        val, Z = c.dense_eigh(A, m=600, B=B)             # products of 6e7 flops and more
        assert np.abs(A @ Z - B @ Z * val).max() < 1e-9
        c.set_initial_states(fi.raw_start_block(w.nbands, c.npw, 17), damp=True)
        assert c.solve(w.e_ref, w.nstates, tol=1e-6)["nconv"] == w.nstates
        loss, rows = c.precond_train(w.e_ref, w.nstates, tol=1e-4, epochs=2)
        assert rows > 0 and np.isfinite(loss)

use()
use()
rt = ctypes.CDLL("libcudart.so.13")
for size in (1024, 4096, 1 << 20):
    assert rt.cudaDeviceReset() == 0
    other = ctypes.c_void_p()                            # may come to lie where the page was
    assert rt.cudaHostAlloc(ctypes.byref(other), ctypes.c_size_t(size), 0) == 0
    use()
    assert not any(ctypes.string_at(other, size))        # nobody wrote into it
print("every context worked")
"""


def test_context_after_a_device_reset():
    env = dict(os.environ, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "every context worked" in r.stdout, r.stdout + r.stderr


@pytest.fixture(scope="module")
def fs():
    from paper_1907_06821_gb300 import build as b
    b.build()
    import paper_1907_06821_gb300 as m
    return m


def _make(fs):
    return fs.Context((10.0, 10.0, 10.0), (16, 16, 16), 3.0, (0, 0, 0), np.zeros((16, 16, 16)))


def _median_us(fs, n=40):
    t = []
    for _ in range(n):
        t0 = time.perf_counter()
        _make(fs).close()
        t.append(time.perf_counter() - t0)
    return 1e6 * float(np.median(t))


def test_one_context_at_a_time(fs):
    """Making and destroying the only context costs less than 2.4 times what it costs beside another
    one (device memory of the last context goes back to the driver, 1.8 times; with a page pinned and
    unpinned each time it was 3.3 times)."""
    torch = pytest.importorskip("torch")
    torch.zeros(1, device="cuda")
    _median_us(fs, 5)
    ratio = []
    for _ in range(3):                                   # (the best of three: the host is shared)
        alone = _median_us(fs)
        with _make(fs):
            beside = _median_us(fs)
        ratio.append(alone / beside)
    assert min(ratio) < 2.4


def test_more_contexts_than_a_page_holds(fs):
    """300 contexts at once (255 flags a page), destroyed in mixed order, each with its own flag."""
    rng = np.random.default_rng(2)
    c = [_make(fs) for _ in range(300)]
    for i in (0, 17, 254, 255, 299):
        c[i].wait_selftest(64, pending=True)
    for i in (0, 17, 254, 255, 299):
        c[(i + 5) % 300].spectral_bounds(3)              # the neighbour's flag is not raised
        with pytest.raises(fs.FSError) as ei:
            c[i].spectral_bounds(3)
        assert ei.value.code == fs.FS_ERR_TIMEOUT
    for i in rng.permutation(300)[:299]:
        c[i].close()
    more = [_make(fs) for _ in range(10)]
    for k in more:
        k.spectral_bounds(3)
        k.close()
