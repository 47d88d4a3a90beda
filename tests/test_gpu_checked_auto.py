"""The checked build (-DMD_CHECKED, as in test_gpu_checked) on the steps that a
context takes by its size and on the field calls: the small step with one and
several clusters, each pair once with blocks of 1024 and 1536 records, a scan,
diagnosed steps, detectors, image forces, uncharged records, and both stateless
field calls at ragged sizes.  No bounds error, and the bits of the normal build."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCENARIO = r"""
import hashlib, sys
import numpy as np
import torch
sys.path.insert(0, sys.argv[1])
from paper_1307_3711_gb300 import md, synth
h = hashlib.sha256()
def feed(g):
    for k in ("x", "u", "z", "kind"):
        h.update(np.ascontiguousarray(getattr(g, k)).tobytes())
def records(n, dark=0, L=0.05):
    rng = np.random.default_rng(n)
    z = np.where(np.arange(n) < n // 4, 3, -1)
    kind = np.where(z < 0, md.KIND_ELECTRON, md.KIND_ION).astype(np.uint8)
    if dark:
        z[n // 2:n // 2 + dark] = 0
        kind[n // 2:n // 2 + dark] = md.KIND_INACTIVE
    u = rng.normal(size=(n, 3)) * 4e-3
    u[z == 0] = 0.0
    return md.HostParticles(rng.uniform(-0.5 * L, 0.5 * L, (n, 3)), u, z.astype(np.int32),
                            np.where(z < 0, 1.0, 5000.0), np.ones(n), kind)
def cfg(**kw):
    return md.make_config(a0=0.01, tau=1.0, dt=0.02, softening=1e-3, envelope=synth.ENV_FLAT, **kw)
def run(sizes, auto=True, det=False, dark=0, **kw):
    with md.Context([cfg(**kw)] * len(sizes), [records(n, dark) for n in sizes]) as ctx:
        assert (ctx.tuning()[4] == md.JSPLIT_AUTO) == auto, sizes
        if det:
            ctx.set_detectors(len(sizes) - 1, 0.03, e_max_ev=500.0, n_bins=16)
        ctx.step(19)                       # a graph replay and direct steps
        if not det and not kw.get("min_image"):
            for d in ctx.step_diag():
                h.update(np.array([d["ke"], d["pe"], d["n_active"]]).tobytes())
        else:
            for k in range(len(sizes)):
                d = ctx.diagnostics(k)
                h.update(np.array([d["ke"], d["pe"], d["n_active"]]).tobytes())
        ctx.sync()
        for k in range(len(sizes)):
            feed(ctx.get_particles(k))
        if det:
            det, ins = ctx.iedf(len(sizes) - 1)
            h.update(det.tobytes()); h.update(ins.tobytes())
            assert det[4].sum() > 0
run([1]); run([5000]); run([4097], det=True)
run([700, 1, 3001, 1040])                  # several clusters in the small step
run([5000], dark=1500)
for n in (9300, 12305):                    # each pair once, blocks of 1024
    run([n])
run([12000], det=True); run([12305], dark=5000)
run([41003]); run([41003], det=True); run([46000], dark=9000)   # blocks of 1536
run([5000, 9300, 33, 12345, 1025])         # a scan
run([11000], boundary=1, box=0.05, min_image=1)
run([11280], boundary=1, box=0.05, min_image=1)
run([12304, 11008], boundary=2, box=0.05, t_switch=0.2, min_image=1, det=True)
run([3000], auto=False, boundary=1, box=0.05, min_image=1)
st = torch.cuda.current_stream().cuda_stream
rng = np.random.default_rng(0)
for nt, ns in ((1, 1), (7, 999), (305, 8003), (300, 70001), (609, 35000), (1217, 1023), (9000, 513),
               (9000, 62), (32768, 360), (8193, 8192), (14001, 8200), (28001, 8195), (100003, 520),
               (300, 12001), (3000, 100007)):
    src = torch.from_numpy(rng.normal(size=(ns, 4)).astype(np.float32)).cuda()
    tgt = torch.from_numpy(rng.normal(size=(nt, 4)).astype(np.float32)).cuda()
    for f in (md.coulomb_field_device, md.coulomb_field_device_noalloc):
        if nt > 32768 and f is md.coulomb_field_device_noalloc:
            continue
        for pot in (False, True):
            e = torch.zeros((nt, 3), dtype=torch.float64, device="cuda")
            phi = torch.zeros(nt, dtype=torch.float64, device="cuda")
            f(src.data_ptr(), ns, tgt.data_ptr(), nt, 1e-6, -1, e.data_ptr(),
              phi.data_ptr() if pot else None, st)
            assert md.field_device_status(st) == md.MD_OK, (nt, ns)
            h.update(e.cpu().numpy().tobytes()); h.update(phi.cpu().numpy().tobytes())
print("DIGEST", h.hexdigest())
"""


def _run(env_extra):
    env = dict(os.environ, **env_extra)
    r = subprocess.run([sys.executable, "-c", SCENARIO, ROOT], capture_output=True, text=True,
                       timeout=600, env=env, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-3000:]
    return [ln for ln in r.stdout.splitlines() if ln.startswith("DIGEST")][0]


def test_steps_chosen_by_size_and_field_calls_stay_in_bounds():
    from paper_1307_3711_gb300 import build
    build.build()
    build.build(checked=True)
    checked = _run({"MD_CHECKED": "1"})
    plain = _run({"MD_CHECKED": "0"})
    assert checked == plain
