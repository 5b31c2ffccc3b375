"""Calls on a nearly full device: FP64 products make digit images of the projector table and of
their operands where there is room, and do without them where there is none."""
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


class Ballast:
    """Holds all device memory but `leave` bytes."""

    def __init__(self, leave):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        self.held = torch.empty(max(0, free - leave), dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *a):
        del self.held
        torch.cuda.empty_cache()


def _bands(c, n, seed):
    x = torch.as_tensor(fi.raw_start_block(n, c.npw, seed), device="cuda")
    torch.cuda.synchronize()
    return x


# 512 projectors x 41,657 plane waves: 0.60 GB an image, per-call images of as much.  900 MB free:
# no kept image (more than an eighth), per-call images whole; 300 MB: in chunks; 110 MB (one column
# buffer of 96 MB more than everything else that the call needs): the FMA kernels or small chunks
@pytest.mark.parametrize("leave", [900, 300, 110])
def test_fp64_application_on_a_full_device(fs, leave):
    w = fi.make_medium()
    with fs.Context.from_workload(w, precision=fs.FS_FP64) as c:
        x = _bands(c, 16, 3)
        ref = c.apply_H(x, shift=0.1)
    tiny = fi.make_config("tiny")
    with fs.Context.from_workload(tiny, precision=fs.FS_FP64) as c:  # every kernel is loaded by now
        c.apply_H(_bands(c, 2, 3))
    with fs.Context.from_workload(w, precision=fs.FS_FP64) as c:
        out = torch.empty_like(x)
        with Ballast(leave << 20):
            for _ in range(2):
                c.apply_H(x, out=out, shift=0.1)
                assert (out - ref).abs().max().item() < 1e-12 * ref.abs().max().item()
        c.apply_H(x, out=out, shift=0.1)
        assert (out - ref).abs().max().item() < 1e-12 * ref.abs().max().item()


def test_images_are_given_back(fs):
    """The images of an earlier application (1.2 GB) make room for the blocks of a call that needs
    more than the 300 MB that are free."""
    w = fi.make_medium()
    with fs.Context.from_workload(w, precision=fs.FS_FP64) as c:
        x = _bands(c, 16, 3)
        ref = c.apply_H(x, shift=0.1)
        want = c.chebfd(0.0, 0.3, -12.0, 13.0, 4, 256, 1)["nfound"]
    with fs.Context.from_workload(w, precision=fs.FS_FP64) as c:
        before = torch.cuda.mem_get_info()[0]
        out = c.apply_H(x, shift=0.1)
        assert before - torch.cuda.mem_get_info()[0] > 1 << 30
        with Ballast(300 << 20):
            assert c.chebfd(0.0, 0.3, -12.0, 13.0, 4, 256, 1)["nfound"] == want
            c.apply_H(x, out=out, shift=0.1)
        assert (out - ref).abs().max().item() < 1e-12 * ref.abs().max().item()


def test_images_of_products_are_given_back(fs):
    """The same for the images of an earlier call's operands (0.6 GB; projectors formed where they
    are used have no table to keep an image of)."""
    w = fi.make_medium()
    with fs.Context.from_workload(w, precision=fs.FS_FP64, projectors=fs.FS_PROJ_GENERATED) as c:
        want = c.chebfd(0.0, 0.3, -12.0, 13.0, 4, 160, 1)["nfound"]
    with fs.Context.from_workload(w, precision=fs.FS_FP64, projectors=fs.FS_PROJ_GENERATED) as c:
        x = _bands(c, 16, 3)
        out = c.apply_H(x, shift=0.1)
        ref = out.clone()
        with Ballast(300 << 20):
            assert c.chebfd(0.0, 0.3, -12.0, 13.0, 4, 160, 1)["nfound"] == want
            c.apply_H(x, out=out, shift=0.1)
        assert (out - ref).abs().max().item() < 1e-12 * ref.abs().max().item()
