"""The automatic steps after a device wait that ran out (the self-test's: the
error word is set, reported and cleared): the step has not moved, and the
context then takes the same steps, bit for bit, as one that saw no expired
wait."""
import numpy as np
import pytest

from paper_1307_3711_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def md():
    from paper_1307_3711_gb300 import build
    build.build()
    from paper_1307_3711_gb300 import md as m
    return m


@pytest.mark.parametrize("n", [300, 4097, 8900, 9500, 41000])
def test_steps_go_on_after_an_expired_wait(md, n):
    rng = np.random.default_rng(n)
    z = np.where(np.arange(n) < n // 4, 3, -1).astype(np.int32)
    recs = (rng.uniform(-0.025, 0.025, (n, 3)), rng.normal(size=(n, 3)) * 4e-3, z,
            np.where(z < 0, 1.0, 5000.0), np.ones(n))
    cfg = md.make_config(a0=0.01, tau=1.0, softening=1e-3, envelope=synth.ENV_FLAT)
    out = []
    for expired in (False, True):
        with md.Context([cfg], [md.HostParticles(*recs)]) as ctx:
            ctx.step(3)
            if expired:
                assert ctx.wait_selftest(20.0) == md.MD_ERR_TIMEOUT
            assert ctx.step_index() == 3
            ctx.step(18)
            assert ctx.step_index() == 21
            out.append(ctx.get_particles(0))
    assert np.array_equal(out[0].x, out[1].x) and np.array_equal(out[0].u, out[1].u)
