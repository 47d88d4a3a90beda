"""md_get_tuning and md_set_tuning as a round trip: what one context reports,
set in itself or in another, takes the same kind of step, and the choice by size
can be taken up again after a forced configuration."""
import numpy as np
import pytest

from paper_1307_3711_gb300 import synth

pytestmark = pytest.mark.gpu
FORCED = (128, 4, 512, 0, 0, 0)


@pytest.fixture(scope="module")
def md():
    from paper_1307_3711_gb300 import build
    build.build()
    from paper_1307_3711_gb300 import md as m
    return m


def _context(md, n, **kw):
    rng = np.random.default_rng(n)
    z = np.where(np.arange(n) < n // 4, 3, -1).astype(np.int32)
    cfg = md.make_config(a0=0.01, tau=1.0, softening=1e-3, envelope=synth.ENV_FLAT, **kw)
    return md.Context([cfg], [md.HostParticles(rng.uniform(-0.03, 0.03, (n, 3)),
                                               rng.normal(size=(n, 3)) * 4e-3, z,
                                               np.where(z < 0, 1.0, 5000.0), np.ones(n))])


def _stepped(ctx):
    ctx.step(2)
    return ctx.get_particles(0).u


@pytest.mark.parametrize("n", [300, 12000])
def test_reported_tuning_takes_the_same_step(md, n):
    with _context(md, n) as ctx:
        auto = ctx.tuning()
        assert auto[4] == md.JSPLIT_AUTO
        default = _stepped(ctx)
    with _context(md, n) as ctx:
        ctx.set_tuning(*FORCED)
        forced = ctx.tuning()
        assert forced[4] != md.JSPLIT_AUTO
        by_force = _stepped(ctx)
    assert not np.array_equal(default, by_force)
    for tunings, want in (((auto,), default), ((forced,), by_force),
                          ((FORCED, auto), default), ((auto, forced), by_force)):
        with _context(md, n) as ctx:
            for t in tunings:
                ctx.set_tuning(*t)
            assert (ctx.tuning()[4] == md.JSPLIT_AUTO) == (tunings[-1] == auto)
            assert np.array_equal(_stepped(ctx), want)


def test_choice_by_size_where_it_is_not_taken(md):
    """A sliced context keeps the step kernel, and takes the choice up again
    when the slice is undone; an unknown configuration is refused as before."""
    n = 12000
    with _context(md, n) as ctx:
        auto = ctx.tuning()
        want = _stepped(ctx)
    with _context(md, n) as ctx:
        ctx.set_slice(0, 0, 4096)
        ctx.set_tuning(*auto)
        assert ctx.tuning()[4] != md.JSPLIT_AUTO
        ctx.set_slice(0, 0, n)
        assert ctx.tuning() == auto
        with pytest.raises(md.MDError):
            ctx.set_tuning(33, 4, 512, 0, md.JSPLIT_AUTO, 0)
        with pytest.raises(md.MDError):
            ctx.set_tuning(128, 4, 512, 0, 65, 0)
        assert ctx.tuning() == auto
        assert np.array_equal(_stepped(ctx), want)
