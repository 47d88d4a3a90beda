"""md_get_particles into page-locked arrays that a kernel's stores could not
reach element by element: arrays that start off a multiple of their element's
size, and arrays that run past the end of a registered block.  Both hold the
records that plain arrays receive, and nothing around them changes."""
import mmap

import numpy as np
import pytest

from paper_1307_3711_gb300 import synth

pytestmark = pytest.mark.gpu
FIELDS = (("x", np.float64, 3), ("u", np.float64, 3), ("z", np.int32, 1), ("mass", np.float64, 1),
          ("w", np.float64, 1), ("kind", np.uint8, 1))


@pytest.fixture(scope="module")
def md():
    from paper_1307_3711_gb300 import build
    build.build()
    from paper_1307_3711_gb300 import md as m
    return m


def _context(md, n):
    rng = np.random.default_rng(n)
    z = rng.choice([-1, 2], size=n).astype(np.int32)
    cfg = md.make_config(a0=0.01, tau=1.0, softening=1e-3, envelope=synth.ENV_FLAT)
    return md.Context([cfg], [md.HostParticles(rng.normal(size=(n, 3)) * 0.02,
                                               rng.normal(size=(n, 3)) * 1e-2, z,
                                               np.where(z < 0, 1.0, 5000.0),
                                               rng.uniform(0.5, 2.0, n))])


def _views(buf, n, skew):
    """The six arrays of n records one after the other in buf, each `skew` bytes
    past a multiple of 16; returns them and the mask of the bytes they cover."""
    out, used, at = {}, np.zeros(buf.size, bool), 0
    for name, t, k in FIELDS:
        at = (at + 15) // 16 * 16 + skew
        size = n * k * np.dtype(t).itemsize
        v = buf[at:at + size].view(t)
        out[name] = v.reshape(n, 3) if k == 3 else v
        used[at:at + size] = True
        at += size
    return out, used


def _get_into(md, ctx, arrays):
    p = md.HostParticles.empty(ctx.sizes[0])
    for name, v in arrays.items():
        setattr(p, name, v)
    ctx.get_particles(0, p)


def _check(md, ctx, buf, n, skew):
    want = ctx.get_particles(0)
    buf[:] = 0xA5
    arrays, used = _views(buf, n, skew)
    _get_into(md, ctx, arrays)
    for name, _, _ in FIELDS:
        assert np.array_equal(arrays[name], getattr(want, name)), name
    assert (buf[~used] == 0xA5).all()


@pytest.mark.parametrize("skew", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("n", [1, 33, 1000])
def test_arrays_at_any_byte_of_a_pinned_buffer(md, n, skew):
    import torch
    buf = torch.zeros(70 * n + 200, dtype=torch.uint8, pin_memory=True).numpy()
    with _context(md, n) as ctx:
        ctx.step(2)
        _check(md, ctx, buf, n, skew)


@pytest.mark.parametrize("pages", [1, 3, 7])
def test_arrays_past_the_end_of_a_registered_block(md, pages):
    import torch
    mem = mmap.mmap(-1, 8 * mmap.PAGESIZE)
    buf = np.frombuffer(mem, dtype=np.uint8)
    n = buf.size // 70
    rt = torch.cuda.cudart()
    with _context(md, n) as ctx:
        ctx.step(2)
        assert int(rt.cudaHostRegister(buf.ctypes.data, pages * mmap.PAGESIZE, 0)) == 0
        try:
            _check(md, ctx, buf, n, 0)
        finally:
            assert int(rt.cudaHostUnregister(buf.ctypes.data)) == 0
