"""The step that evaluates each pair once with records that carry no charge
(unused slots, neutral atoms, test particles of no weight) in whole tiles, whole
blocks and beside charged ones: kicks and diagnostics against the FP64 oracle
and the step kernel; slots beyond the range of FP32 disturb no one."""
import os

import numpy as np
import pytest

import oracle
from paper_1307_3711_gb300 import synth
from tests.helpers import force_error, summary

pytestmark = pytest.mark.gpu
FORCE_P99 = 2e-5     # the force gate of the other field and step tests
DT = 0.02
EPS = 1e-3
NTHREADS = os.cpu_count() or 1
FORCED = (128, 4, 512, 0, 0, 0)


@pytest.fixture(scope="module")
def md():
    from paper_1307_3711_gb300 import build
    build.build()
    from paper_1307_3711_gb300 import md as m
    return m


def _uncharged(n, where):
    """Mask of the uncharged records."""
    k = np.arange(n)
    block = 1536 if n >= 40000 else 1024
    return {"last": k >= n // 2, "first": k < n // 2, "last_tile": k >= n - 100,
            "middle": (k >= block + 100) & (k < 4 * block + 70),
            "blocks": (k // block) % 2 == 1, "tiles": (k // 128) % 2 == 0,
            "scattered": np.random.default_rng(n).random(n) < 0.5, "all": k >= 0}[where]


def _records(n, where, what, md, L=0.05):
    rng = np.random.default_rng(n + len(where))
    off = _uncharged(n, where)
    x = rng.uniform(-0.5 * L, 0.5 * L, (n, 3))
    u = rng.normal(size=(n, 3)) * 4e-3
    z = np.where(np.arange(n) % 7 < 2, 3, -1)
    w = np.ones(n)
    kind = np.where(z < 0, md.KIND_ELECTRON, md.KIND_ION).astype(np.uint8)
    if what == "slots":
        z[off], kind[off], u[off] = 0, md.KIND_INACTIVE, 0.0
    elif what == "neutral":
        z[off], kind[off] = 0, md.KIND_ION
    else:                      # test particles: their charge moves them, and no one else
        w[off] = 0.0
    return x, u, z.astype(np.int32), np.where(z < 0, 1.0, 5000.0), w, kind


def _cfg(md, **kw):
    return md.make_config(a0=0.0, tau=1.0, dt=DT, softening=EPS, envelope=synth.ENV_FLAT, **kw)


@pytest.mark.parametrize("what", ["slots", "neutral", "test"])
@pytest.mark.parametrize("n,where", [
    (9300, "last"), (9300, "first"), (9300, "blocks"), (9300, "all"), (12305, "last_tile"),
    (12305, "middle"), (12305, "tiles"), (12305, "scattered"), (40100, "last"),
    (40100, "blocks"), (40100, "middle")])
def test_kicks_and_diagnostics(md, n, where, what):
    recs = _records(n, where, what, md)
    x, u, z, mass, w, kind = recs
    got = {}
    for name, forced, diag in (("auto", None, False), ("diag", None, True), ("step", FORCED, True)):
        with md.Context([_cfg(md)], [md.HostParticles(*recs)]) as ctx:
            if forced:
                ctx.set_tuning(*forced)
            d = ctx.step_diag()[0] if diag else ctx.step(1)
            got[name] = (ctx.get_particles(0), d)
    assert np.array_equal(got["auto"][0].u, got["diag"][0].u)
    assert np.array_equal(got["auto"][0].x, got["diag"][0].x)
    g = got["auto"][0]
    still = z == 0
    assert np.array_equal(g.u[still], u[still])
    idx = np.flatnonzero(~still)
    if len(idx) > 400:
        idx = np.unique(np.r_[idx[:3], idx[-3:],
                              np.random.default_rng(1).choice(idx, 400, replace=False)])
    q = w * z
    if len(idx) and q.any():
        kick = (g.u[idx] - u[idx]) * (mass[idx] / (z[idx] * DT))[:, None]
        e64 = oracle.coulomb_field(x[idx], x, q, EPS, oracle.coulomb_constant(0.8), self_idx=idx,
                                   nthreads=NTHREADS)
        assert summary(force_error(kick, e64))["p99"] <= FORCE_P99
    elif len(idx):
        assert np.array_equal(g.u, u)
    d, d0 = got["diag"][1], got["step"][1]
    scale = abs(d0["pe"]) + d0["ke"]
    for k in ("ke", "pe", "total"):
        assert abs(d[k] - d0[k]) <= 1e-6 * scale
    assert d["n_active"] == d0["n_active"] and np.array_equal(d["charge_count"],
                                                              d0["charge_count"])


@pytest.mark.parametrize("n,where", [(12288, "last"), (11296, "first"), (12305, "tiles")])
def test_minimum_image_kicks(md, n, where):
    L = 0.05
    x, u, z, mass, w, kind = recs = _records(n, where, "slots", md, L)
    with md.Context([_cfg(md, boundary=1, box=L, min_image=1)], [md.HostParticles(*recs)]) as ctx:
        ctx.step(1)
        g = ctx.get_particles(0)
    idx = np.random.default_rng(2).choice(np.flatnonzero(z), 400, replace=False)
    kick = (g.u[idx] - u[idx]) * (mass[idx] / (z[idx] * DT))[:, None]
    e64 = oracle.coulomb_field(x[idx], x, w * z, EPS, oracle.coulomb_constant(0.8), self_idx=idx,
                               box=L, nthreads=NTHREADS)
    assert summary(force_error(kick, e64))["p99"] <= FORCE_P99


@pytest.mark.parametrize("n,at", [(12288, 6144), (46080, 30720)])
def test_slots_out_of_range_disturb_no_one(md, n, at):
    """Unused slots in tiles and blocks of their own at positions that FP32 cannot
    hold: the charged records move as without them."""
    rng = np.random.default_rng(n)
    x = rng.uniform(-0.02, 0.02, (n, 3))
    x[at:] = 1e39
    u = rng.normal(size=(n, 3)) * 4e-3
    u[at:] = 0.0
    z = np.where(np.arange(n) % 7 < 2, 3, -1)
    z[at:] = 0
    kind = np.where(z < 0, md.KIND_ELECTRON, md.KIND_ION).astype(np.uint8)
    kind[at:] = md.KIND_INACTIVE
    recs = (x, u, z.astype(np.int32), np.where(z < 0, 1.0, 5000.0), np.ones(n), kind)
    with md.Context([_cfg(md)], [md.HostParticles(*recs)]) as ctx:
        ctx.step(3)
        g = ctx.get_particles(0)
    with md.Context([_cfg(md)], [md.HostParticles(*(a[:at] for a in recs))]) as ctx:
        ctx.step(3)
        want = ctx.get_particles(0)
    assert np.isfinite(g.u[:at]).all()
    scale = np.abs(want.u - u[:at]).max()
    assert np.abs(g.u[:at] - want.u).max() <= 1e-5 * scale


@pytest.mark.parametrize("n,charged,chosen", [(60000, 1.0, True), (60000, 0.4, True),
                                              (60000, 0.3, False), (60000, 0.0, False),
                                              (30000, 0.1, True)])
def test_large_contexts_of_slots_keep_the_step_kernel(md, n, charged, chosen):
    x, u, z, mass, w, kind = _records(n, "last", "charged", md)
    w = np.ones(n)
    off = np.arange(n) >= charged * n
    z[off], kind[off], u[off], mass[off] = 0, md.KIND_INACTIVE, 0.0, 1.0
    with md.Context([_cfg(md)], [md.HostParticles(x, u, z, mass, w, kind)]) as ctx:
        assert (ctx.tuning()[4] == md.JSPLIT_AUTO) == chosen
        ctx.step(1)
        g = ctx.get_particles(0)
    assert np.array_equal(g.x[off], x[off])
    if charged:
        idx = np.random.default_rng(3).choice(np.flatnonzero(z), 300, replace=False)
        kick = (g.u[idx] - u[idx]) * (mass[idx] / (z[idx] * DT))[:, None]
        e64 = oracle.coulomb_field(x[idx], x, (w * z).astype(float), EPS,
                                   oracle.coulomb_constant(0.8), self_idx=idx, nthreads=NTHREADS)
        assert summary(force_error(kick, e64))["p99"] <= FORCE_P99


def test_charged_records_set_later_take_the_choice_up(md):
    """A large context made of neutral atoms keeps the step kernel until
    md_set_particles gives it charges, and a forced tuning beyond that."""
    n = 41000
    recs = _records(n, "last", "charged", md)
    x, u, z, mass, w, kind = recs
    w = np.ones(n)
    neutral = (x, u, np.zeros(n, np.int32), mass, w, np.zeros(n, np.uint8))
    charged = (x, u, z, mass, w, kind)
    for forced in (False, True):
        with md.Context([_cfg(md)], [md.HostParticles(*neutral)]) as ctx:
            assert ctx.tuning()[4] != md.JSPLIT_AUTO
            ctx.step(2)
            if forced:
                ctx.set_tuning(*FORCED)
            ctx.set_particles(0, md.HostParticles(*neutral))
            assert ctx.tuning()[4] != md.JSPLIT_AUTO
            ctx.set_particles(0, md.HostParticles(*charged))
            assert (ctx.tuning()[4] == md.JSPLIT_AUTO) != forced
            ctx.step(1)
            got = ctx.get_particles(0).u
        with md.Context([_cfg(md)], [md.HostParticles(*charged)]) as ctx:
            if forced:
                ctx.set_tuning(*FORCED)
            ctx.step(1)
            assert np.array_equal(ctx.get_particles(0).u, got)
