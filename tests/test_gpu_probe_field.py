"""The single-launch field evaluation (clusters of CTAs that add their partial
sums on the chip; a plain kernel for few sources): target counts around its
groups, source counts around its slices, stages and cluster sizes, both
stateless entry points and a context's field, against the FP64 oracle."""
import os

import numpy as np
import pytest

import oracle
from paper_1307_3711_gb300 import synth
from tests.helpers import force_error, summary

pytestmark = pytest.mark.gpu
FORCE_P99 = 2e-5     # the force gate of the other field tests
EPS = 1e-3
NTHREADS = os.cpu_count() or 1


@pytest.fixture(scope="module")
def md():
    from paper_1307_3711_gb300 import build
    build.build()
    from paper_1307_3711_gb300 import md as m
    return m


@pytest.mark.parametrize("alloc", [True, False])
@pytest.mark.parametrize("nt,ns", [(1, 1), (1, 16000), (4, 15), (7, 999), (33, 2000), (65, 3999),
                                   (305, 8003), (1217, 1023), (2500, 16385), (3071, 3073),
                                   (8193, 511), (9000, 1), (9000, 513), (32768, 40), (1500, 100),
                                   (8193, 8192), (20000, 9001)])
def test_field_and_potential_follow_oracle(md, nt, ns, alloc):
    import torch
    rng = np.random.default_rng(nt * 7 + ns)
    kc = oracle.coulomb_constant(0.8)
    xs = (rng.normal(size=(ns, 3)) * 0.02).astype(np.float32)
    xt = (rng.normal(size=(nt, 3)) * 0.02).astype(np.float32)
    qs = rng.choice([-1.0, 1.0, 3.0], size=ns)
    src = torch.tensor(np.c_[xs, kc * qs], dtype=torch.float32, device="cuda")
    tgt = torch.tensor(np.c_[xt, np.zeros(nt)], dtype=torch.float32, device="cuda")
    f = md.coulomb_field_device if alloc else md.coulomb_field_device_noalloc
    st = torch.cuda.current_stream().cuda_stream
    got = []
    for pot in (True, False, True):
        e = torch.full((nt, 3), float("nan"), dtype=torch.float64, device="cuda")
        phi = torch.full((nt,), float("nan"), dtype=torch.float64, device="cuda")
        f(src.data_ptr(), ns, tgt.data_ptr(), nt, EPS * EPS, -1, e.data_ptr(),
          phi.data_ptr() if pot else None, st)
        torch.cuda.synchronize()
        got.append((e.cpu().numpy(), phi.cpu().numpy()))
    assert md.field_device_status(st) == md.MD_OK
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][0], got[2][0])
    assert np.array_equal(got[0][1], got[2][1]) and np.isnan(got[1][1]).all()
    e64, p64 = oracle.coulomb_field(xt.astype(float), xs.astype(float), qs, EPS, kc,
                                    potential=True, nthreads=NTHREADS)
    assert summary(force_error(got[0][0], e64))["p99"] <= FORCE_P99
    np.testing.assert_allclose(got[0][1], p64, rtol=1e-5, atol=1e-5 * np.abs(p64).max())


@pytest.mark.parametrize("n", [1, 17, 2000, 4099])
def test_small_contexts_field_follows_oracle(md, n):
    """md_get_fields of a small context: its records are targets and sources
    (the potential without their own term)."""
    rng = np.random.default_rng(n)
    x = rng.normal(size=(n, 3)) * 0.02
    z = rng.choice([-1, 1, 3], size=n).astype(np.int32)
    cfg = md.make_config(a0=0.0, tau=1.0, softening=EPS, envelope=synth.ENV_FLAT)
    with md.Context([cfg], [md.HostParticles(x, x * 0, z, np.ones(n), np.ones(n))]) as ctx:
        e, phi = ctx.fields(0, potential=True)
    e64, p64 = oracle.self_field(x, z.astype(float), EPS, oracle.coulomb_constant(0.8),
                                 potential=True, nthreads=NTHREADS)
    if n > 1:
        assert summary(force_error(e, e64))["p99"] <= FORCE_P99
    np.testing.assert_allclose(phi, p64, rtol=1e-4, atol=2e-5 * max(np.abs(p64).max(), 1e-7))


@pytest.mark.parametrize("nt,ns", [(1, 12000), (32, 66001), (33, 12001), (74, 150007), (75, 40000),
                                   (148, 99999), (149, 12000), (304, 70001), (305, 13000),
                                   (457, 61000), (608, 35000), (609, 35000)])
def test_large_tiles_follow_oracle(md, nt, ns):
    """Few targets of many sources: the target counts at which the split changes,
    source counts of one to several stages per CTA with ragged ends."""
    test_field_and_potential_follow_oracle(md, nt, ns, False)


@pytest.mark.parametrize("nt,ns", [(1500, 62), (1500, 63), (32768, 360), (32768, 361), (256, 1),
                                   (30000, 300)])
def test_few_sources_follow_oracle(md, nt, ns):
    """Either side of the line between the kernel for few sources and the clusters."""
    test_field_and_potential_follow_oracle(md, nt, ns, False)
