"""The ionization pass's field at the ions when its kernel takes a tile of
sources per CTA and the segments are formed from the tiles' sums: clusters of
one tile and a few records, of exactly as many tiles as the scratch holds and of
one more (the segments summed by the kernel itself), with a live region that ends
inside a tile, against the FP64 oracle."""
import os

import numpy as np
import pytest

import oracle
from paper_1307_3711_gb300 import synth

pytestmark = pytest.mark.gpu
AR = synth.ARGON
NTHREADS = os.cpu_count() or 1


@pytest.fixture(scope="module")
def md():
    from paper_1307_3711_gb300 import build
    build.build()
    from paper_1307_3711_gb300 import md as m
    return m


@pytest.mark.parametrize("atoms,mean_z", [(57, 1), (57, 8), (1000, 0), (3000, 3), (6371, 8),
                                          (6372, 8)])
def test_pass_field_follows_oracle(md, atoms, mean_z):
    zmax = 8
    rng = np.random.default_rng(atoms + mean_z)
    c = synth.make_cluster(3, atoms, 0, synth.nm_to_len(8.0 * (atoms / 2e5) ** (1 / 3)), 0,
                           AR["mass"], n_electron_slots=atoms * zmax)
    z = np.zeros(c.n, dtype=np.int32)
    z[:atoms] = zmax if mean_z == zmax else rng.binomial(zmax, mean_z / zmax, size=atoms)
    # the freed electrons fill the slots densely, each near an ion
    free = int(z[:atoms].sum())
    kind = np.full(c.n, md.KIND_INACTIVE, dtype=np.uint8)
    kind[:atoms] = md.KIND_ION
    kind[atoms:atoms + free] = md.KIND_ELECTRON
    x, mass = c.x.copy(), np.where(np.arange(c.n) < atoms, AR["mass"], 1.0)
    host = np.repeat(np.arange(atoms), z[:atoms])
    x[atoms:atoms + free] = x[host] + rng.normal(size=(free, 3)) * synth.nm_to_len(0.3)
    z[atoms:atoms + free] = -1
    rw = synth.nm_to_len(AR["r_w_nm"])
    eps = synth.nm_to_len(0.1)
    cfg = md.make_config(a0=0.0, tau=1.0, dt=0.02, softening=eps, envelope=3, rate_model=1,
                         ionize_every=0, zmax=zmax, n_ions=atoms, slot_base=atoms, seed=5,
                         r_loc=3 * rw, r_create=rw, species=AR)
    hp = md.HostParticles(x, np.zeros_like(x), z, mass, c.w, kind)
    with md.Context([cfg], [hp]) as ctx:
        ctx.ionize()
        emag = ctx.ionization(0)["emag"]
    live = kind != md.KIND_INACTIVE
    q = np.where(live, c.w * z, 0.0)
    e64 = oracle.coulomb_field(x[:atoms], x[live], q[live], eps, oracle.coulomb_constant(0.8),
                               self_idx=np.arange(atoms), nthreads=NTHREADS)
    emag64 = np.linalg.norm(e64, axis=1)
    # FP32 pair terms, compensated: the force gate of the other field tests
    rel = np.abs(emag - emag64) / max(np.sqrt(np.mean(emag64 ** 2)), 1e-300)
    assert np.percentile(rel, 99) < 2e-5
