"""Ion energy detectors with the steps that a context takes by its size: the
push of the step that evaluates each pair once (with eight and with four warps a
group, and with image forces) and of the small step record every crossing that
the oracle's detectors find in the GPU's own states."""
import math

import numpy as np
import pytest

import oracle
from paper_1307_3711_gb300 import synth

pytestmark = pytest.mark.gpu
KC = oracle.coulomb_constant(0.8)
ME_C2_EV = 510998.95


@pytest.fixture(scope="module")
def md():
    from paper_1307_3711_gb300 import build
    build.build()
    from paper_1307_3711_gb300 import md as m
    return m


@pytest.mark.parametrize("n,image", [(2500, False), (9600, False), (12305, False), (41000, False),
                                     (12304, True)])
def test_counts_match_oracle_on_gpu_states(md, n, image):
    r0 = synth.nm_to_len(2.0)
    c = synth.make_cluster(n, n, 0, r0, 1, synth.MASS_40AMU)
    q = c.w * c.z
    tau = math.sqrt(synth.MASS_40AMU * r0 ** 3 / (KC * q.sum()))
    e_max_ev = 0.3 * KC * q.sum() / r0 * ME_C2_EV
    kw = dict(boundary=1, box=6.0 * r0, min_image=1) if image else {}
    cfg = md.make_config(a0=0.0, dt=tau / 20, softening=synth.nm_to_len(0.005),
                         envelope=synth.ENV_FLAT, **kw)
    nb, radius = 24, 1.4 * r0
    det = oracle.Detectors(n, radius=radius, cone_deg=30.0, e_max_ev=e_max_ev, nbins=nb)
    with md.Context([cfg], [md.HostParticles.from_cluster(c)]) as ctx:
        ctx.set_detectors(0, radius, cone_deg=30.0, e_max_ev=e_max_ev, n_bins=nb)
        assert ctx.tuning()[4] == md.JSPLIT_AUTO
        g0 = ctx.get_particles(0)
        for _ in range(45):
            ctx.step(1)
            g1 = ctx.get_particles(0)
            det.record(g0.x, g1.x, oracle.State(g1.x, g1.u, g1.z, g1.mass, g1.w,
                                                (g1.kind != 2).astype(np.uint8)))
            g0 = g1
        got, inside = ctx.iedf(0)
    assert n // 10 < det.hist[4].sum() < n and all(det.hist[k].sum() > 0 for k in range(4))
    np.testing.assert_array_equal(got, det.hist)
    np.testing.assert_array_equal(inside, det.inside(oracle.State(
        g0.x, g0.u, g0.z, g0.mass, g0.w, (g0.kind != 2).astype(np.uint8))))
