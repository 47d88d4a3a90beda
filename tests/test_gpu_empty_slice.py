"""An empty target slice (a rank beyond the last block of a split cluster): its
field, diagnostics and steps are those of no record."""
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


@pytest.mark.parametrize("n,at", [(2500, 0), (2500, 1024), (2500, 2500), (12000, 12000)])
def test_empty_slice_has_no_field_and_no_energy(md, n, at):
    rng = np.random.default_rng(n)
    z = rng.choice([-1, 2], size=n).astype(np.int32)
    recs = (rng.normal(size=(n, 3)) * 0.02, rng.normal(size=(n, 3)) * 1e-2, z,
            np.where(z < 0, 1.0, 5000.0), np.ones(n))
    cfg = md.make_config(a0=0.01, tau=1.0, softening=1e-3, envelope=synth.ENV_FLAT)
    with md.Context([cfg], [md.HostParticles(*recs)]) as ctx:
        ctx.set_slice(0, at, at)
        e, phi = ctx.fields(0, potential=True)
        assert not e.any() and not phi.any()
        for d in (ctx.diagnostics(0), ctx.step_diag()[0]):
            assert d["n_active"] == 0 and d["n_nonfinite"] == 0
            assert d["ke"] == d["pe"] == d["total"] == 0.0 and not d["p"].any()
            assert not d["charge_count"].any()
        ctx.step(2)
        assert ctx.step_index() == 3
        g = ctx.get_particles(0)
        assert np.array_equal(g.x, recs[0]) and np.array_equal(g.u, recs[1])
