"""Which contexts take the step chosen for their size: those for which it is the
faster one.  Scans of many clusters of a few hundred records keep the step
kernel, whose blocks they fill better; every choice gives the oracle's kicks."""
import os

import numpy as np
import pytest

import oracle
from paper_1307_3711_gb300 import synth
from tests.helpers import force_error, summary

pytestmark = pytest.mark.gpu
FORCE_P99 = 2e-5     # the force gate of the other field and step tests
DT = 0.02
NTHREADS = os.cpu_count() or 1


@pytest.fixture(scope="module")
def md():
    from paper_1307_3711_gb300 import build
    build.build()
    from paper_1307_3711_gb300 import md as m
    return m


def _records(n, seed):
    rng = np.random.default_rng(seed)
    z = np.where(np.arange(n) < n // 4, 3, -1).astype(np.int32)
    return (rng.uniform(-0.025, 0.025, (n, 3)), rng.normal(size=(n, 3)) * 4e-3, z,
            np.where(z < 0, 1.0, 5000.0), np.ones(n))


@pytest.mark.parametrize("sizes,chosen", [
    ([1], True), ([8990], True), ([9100], True), ([30] * 50, True), ([800] * 100, True),
    ([2500] * 64, True), ([1100] * 200, True), ([300] * 700, False), ([100] * 5000, False),
    ([300] * 1000, False), ([150] * 4000, False), ([150] * 3000 + [41000], False),
    ([12000] + [500] * 20, True)])
def test_choice_is_the_faster_step(md, sizes, chosen):
    recs = {n: _records(n, n) for n in set(sizes)}
    cfg = md.make_config(a0=0.0, tau=1.0, dt=DT, softening=1e-3, envelope=synth.ENV_FLAT)
    with md.Context([cfg] * len(sizes), [md.HostParticles(*recs[n]) for n in sizes]) as ctx:
        assert (ctx.tuning()[4] == md.JSPLIT_AUTO) == chosen
        ctx.step(1)
        for k in {0, len(sizes) // 2, len(sizes) - 1}:
            n = sizes[k]
            x, u, z, mass, w = recs[n]
            got = (ctx.get_particles(k).u - u) * (mass / (z * DT))[:, None]
            idx = np.unique(np.random.default_rng(k).integers(0, n, 300))
            e64 = oracle.coulomb_field(x[idx], x, z.astype(float), 1e-3,
                                       oracle.coulomb_constant(0.8), self_idx=idx,
                                       nthreads=NTHREADS)
            if n > 1:
                assert summary(force_error(got[idx], e64))["p99"] <= FORCE_P99
            else:
                assert not got.any()
