"""Minimum-image forces with each pair evaluated once: record counts that leave
a chunk of 16 sources (padded with sources far away, which an image would bring
near), one and many charges, the mixed boundary on either side of its switch,
several clusters of one context, against the FP64 oracle."""
import os

import numpy as np
import pytest

import oracle
from paper_1307_3711_gb300 import synth
from tests.helpers import force_error, summary

pytestmark = pytest.mark.gpu
FORCE_P99 = 2e-5     # the force gate of the other field and step tests
DT, EPS, L = 0.02, 1e-3, 0.05
NTHREADS = os.cpu_count() or 1


@pytest.fixture(scope="module")
def md():
    from paper_1307_3711_gb300 import build
    build.build()
    from paper_1307_3711_gb300 import md as m
    return m


def _records(n, charges, seed):
    rng = np.random.default_rng(seed)
    x = rng.uniform(-0.5 * L, 0.5 * L, (n, 3))
    u = rng.normal(size=(n, 3)) * 1e-4
    z = {"one": np.full(n, 2), "species": np.where(np.arange(n) < n // 4, 3, -1),
         "mixed": rng.integers(-1, 4, n)}[charges]
    w = rng.uniform(0.5, 3.0, n) if charges == "mixed" else np.ones(n)
    return x, u, z.astype(np.int32), np.where(z < 0, 1.0, 5000.0), w


def _check(recs, u, box, n=400):
    x, u0, z, mass, w = recs
    idx = np.random.default_rng(3).choice(np.flatnonzero(z), min(n, np.count_nonzero(z)),
                                          replace=False)
    kick = (u[idx] - u0[idx]) * (mass[idx] / (z[idx] * DT))[:, None]
    e64 = oracle.coulomb_field(x[idx], x, w * z, EPS, oracle.coulomb_constant(0.8), self_idx=idx,
                               box=box, nthreads=NTHREADS)
    assert summary(force_error(kick, e64))["p99"] <= FORCE_P99


def _cfg(md, **kw):
    return md.make_config(a0=0.0, tau=1.0, dt=DT, softening=EPS, envelope=synth.ENV_FLAT, box=L,
                          min_image=1, **kw)


@pytest.mark.parametrize("charges", ["one", "species", "mixed"])
@pytest.mark.parametrize("n", [11280, 12304, 11001])
def test_ragged_chunks(md, n, charges):
    recs = _records(n, charges, n)
    with md.Context([_cfg(md, boundary=1)], [md.HostParticles(*recs)]) as ctx:
        assert ctx.tuning()[4] == md.JSPLIT_AUTO
        ctx.step(1)
        _check(recs, ctx.get_particles(0).u, L)


@pytest.mark.parametrize("n", [11280, 12000])
def test_mixed_boundary_either_side_of_its_switch(md, n):
    """Images before t_switch, none after; the state between is read back."""
    recs = list(_records(n, "species", n + 1))
    with md.Context([_cfg(md, boundary=2, t_switch=1.5 * DT)], [md.HostParticles(*recs)]) as ctx:
        for step, box in ((0, L), (1, L), (2, 0.0), (3, 0.0)):
            ctx.step(1)
            g = ctx.get_particles(0)
            _check(recs, g.u, box)
            recs[0], recs[1] = g.x, g.u


def test_image_and_open_clusters_together(md):
    """Each cluster of a context with and without image forces has its own kicks;
    one small image cluster keeps the step kernel for all of them."""
    for sizes, chosen in (((11280, 12000, 700), True), ((11280, 12000, 700), False)):
        sets = [_records(n, "species", n) for n in sizes]
        cfgs = [_cfg(md, boundary=1),
                md.make_config(a0=0.0, tau=1.0, dt=DT, softening=EPS, envelope=synth.ENV_FLAT),
                _cfg(md, boundary=1) if not chosen else
                md.make_config(a0=0.0, tau=1.0, dt=DT, softening=EPS, envelope=synth.ENV_FLAT)]
        with md.Context(cfgs, [md.HostParticles(*s) for s in sets]) as ctx:
            assert (ctx.tuning()[4] == md.JSPLIT_AUTO) == chosen
            ctx.step(1)
            for k, box in enumerate((L, 0.0, 0.0 if chosen else L)):
                _check(sets[k], ctx.get_particles(k).u, box)
