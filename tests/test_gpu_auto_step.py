"""The steps of contexts whose kernel configuration is not forced (the small
step, and the step that evaluates each pair of records once): record counts
around their target groups, i-blocks, tiles and chunks, one and many charges
per block, several clusters, the diagnostic and the minimum-image twin, against
the FP64 oracle and against the step kernel that sums every pair for either
record."""
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


def _gas(n, charges, seed, L=0.05):
    rng = np.random.default_rng(seed)
    x = rng.uniform(-0.5 * L, 0.5 * L, (n, 3))
    u = rng.normal(size=(n, 3)) * 4e-3
    if charges == "species":       # ions first, then electrons
        z = np.where(np.arange(n) < n // 4, 3, -1)
    elif charges == "one":
        z = np.full(n, 2)
    else:                          # every record its own macro charge, neutrals among them
        z = rng.integers(-1, 4, n)
    w = rng.uniform(0.5, 3.0, n) if charges == "mixed" else np.ones(n)
    mass = np.where(z < 0, 1.0, 5000.0)
    return x, u, z.astype(np.int32), mass, w


def _cfg(md, **kw):
    return md.make_config(a0=0.0, tau=1.0, dt=DT, softening=1e-3, envelope=synth.ENV_FLAT, **kw)


def _kick(md, recs, forced=None, **kw):
    """Momentum increments of one step, in units of the field (du m / (z dt))."""
    x, u, z, mass, w = recs
    with md.Context([_cfg(md, **kw)], [md.HostParticles(x, u, z, mass, w)]) as ctx:
        if forced:
            ctx.set_tuning(*forced)
        ctx.step(1)
        g = ctx.get_particles(0)
    c = z != 0
    return (g.u[c] - u[c]) * (mass[c] / (z[c] * DT))[:, None], c


@pytest.mark.parametrize("charges", ["species", "one", "mixed"])
@pytest.mark.parametrize("n", [1, 2, 16, 17, 33, 1023, 1025, 4095, 4097, 8995, 9217, 10241,
                               11279])
def test_kick_follows_oracle_around_block_and_tile_edges(md, n, charges):
    recs = _gas(n, charges, n)
    x, u, z, mass, w = recs
    got, c = _kick(md, recs)
    e64 = oracle.self_field(x, w * z, 1e-3, oracle.coulomb_constant(0.8), nthreads=NTHREADS)[c]
    if len(got) == 0 or np.abs(e64).max() == 0.0:
        assert np.abs(got).max(initial=0.0) == 0.0
        return
    assert summary(force_error(got, e64))["p99"] <= FORCE_P99
    one, _ = _kick(md, recs, forced=(128, 4, 512, 0, 0, 0))
    assert summary(force_error(got, one))["p99"] <= FORCE_P99


@pytest.mark.parametrize("n", [40000, 46099])
def test_large_blocks_follow_oracle(md, n):
    """From 40000 records on, blocks of 1536 targets."""
    recs = _gas(n, "species", 5)
    x, u, z, mass, w = recs
    got, _ = _kick(md, recs)
    idx = np.r_[0:3, 1534:1538, n - 3:n, np.random.default_rng(1).integers(0, n, 200)]
    q = w * z
    e64 = oracle.coulomb_field(x[idx], x, q, 1e-3, oracle.coulomb_constant(0.8),
                               self_idx=idx, nthreads=NTHREADS)
    assert summary(force_error(got[idx], e64))["p99"] <= FORCE_P99


@pytest.mark.parametrize("largest", [3000, 9600])
def test_clusters_of_one_launch_are_independent(md, largest):
    """Uneven clusters together and alone: the same kicks to FP32 order."""
    sets = [_gas(n, ch, 50 + n) for n, ch in
            ((700, "mixed"), (4100, "species"), (1, "one"), (1040, "one"), (largest, "species"))]
    with md.Context([_cfg(md) for _ in sets], [md.HostParticles(*s) for s in sets]) as ctx:
        ctx.step(1)
        together = [ctx.get_particles(k).u - sets[k][1] for k in range(len(sets))]
    for s, du in zip(sets, together):
        with md.Context([_cfg(md)], [md.HostParticles(*s)]) as ctx:
            ctx.step(1)
            alone = ctx.get_particles(0).u - s[1]
        scale = np.abs(alone).max()
        assert np.abs(du - alone).max() <= 1e-5 * scale


@pytest.mark.parametrize("n,charges", [(1500, "mixed"), (5000, "species"), (9300, "mixed"), (45000, "species")])
def test_diagnostic_step_and_repeats(md, n, charges):
    """md_step_diag takes the same step, bit for bit, as md_step and reports
    the diagnostics at its start; a second context repeats the bits."""
    recs = _gas(n, charges, 9)
    out = []
    for diag in (False, True, False):
        with md.Context([_cfg(md)], [md.HostParticles(*recs)]) as ctx:
            d0 = ctx.diagnostics(0)
            d = ctx.step_diag()[0] if diag else ctx.step(1)
            ctx.step(17)
            out.append((ctx.get_particles(0), d, d0))
    for k in (1, 2):
        assert np.array_equal(out[0][0].x, out[k][0].x)
        assert np.array_equal(out[0][0].u, out[k][0].u)
    d, d0 = out[1][1], out[1][2]
    scale = abs(d0["pe"]) + d0["ke"]
    for k in ("ke", "pe"):
        assert abs(d[k] - d0[k]) <= 1e-6 * scale
    assert np.array_equal(d["charge_count"], d0["charge_count"])


@pytest.mark.parametrize("n", [1000, 4097, 11000, 12305])
def test_minimum_image_kick_follows_oracle(md, n):
    L = 0.05
    recs = _gas(n, "species", n + 3, L)
    x, u, z, mass, w = recs
    got, c = _kick(md, recs, boundary=1, box=L, min_image=1)
    e64 = oracle.self_field(x, w * z, 1e-3, oracle.coulomb_constant(0.8), box=L,
                            nthreads=NTHREADS)[c]
    assert summary(force_error(got, e64))["p99"] <= FORCE_P99
