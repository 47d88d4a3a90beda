"""Surrogate rates at ion counts around the two sizes of a warp's share (16 ions
while they give an SM two CTAs at most, else 32): every ion's rate is the one it has in a
call of another size, bit for bit, and nothing is written past the last ion."""
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


def test_rates_do_not_depend_on_the_number_of_ions(md):
    import torch
    sms, _ = md.device_info()
    line = 128 * sms
    rng = np.random.default_rng(4)
    n = line + 4077
    w = torch.from_numpy(rng.normal(size=5000).astype(np.float32) * 0.1).cuda()
    logu = lambda lo, hi: torch.from_numpy(10.0 ** rng.uniform(lo, hi, n)).cuda()  # noqa: E731
    emag, ne, te = logu(-2.5, -0.3), logu(16, 23), logu(0, 3)
    ne[::7] = 0.0
    emag[::11] = 10.0          # outside the surrogate's domain: the plain rate
    z = torch.from_numpy(rng.integers(-1, 10, n).astype(np.int32)).cuda()
    cfg = md.mlp_train_config(synth.ARGON)
    st = torch.cuda.current_stream().cuda_stream

    def rates(k):
        nu = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        md.ion_rates_device(cfg, md.RATES_MLP, w.data_ptr(), emag.data_ptr(), z.data_ptr(),
                            ne.data_ptr(), te.data_ptr(), k, nu.data_ptr(), st)
        return nu.cpu().numpy()

    want = rates(n)
    assert np.isfinite(want).all()
    for k in (1, 15, 16, 17, 31, 33, 64, 65, 1000, line - 1, line, line + 1, line + 33):
        got = rates(k)
        assert np.array_equal(got[:k], want[:k]), k
        assert np.isnan(got[k:]).all()
