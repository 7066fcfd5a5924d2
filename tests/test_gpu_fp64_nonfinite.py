"""FP64 solves with a sample that holds a NaN or an infinity: T of that sample is NaN
wherever its potential is, on either side of n = 80 (rows of V C formed in the T kernel
or as digit products, which have no digits for such values), the call reports it, and
the other samples keep their bits."""
import numpy as np
import pytest

from paper_2106_00454_gb300 import inputs as W

from parity_util import gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_wp", [24, 39, 48, 100, 150])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_sample(n_wp, bad):
    import torch
    from paper_2106_00454_gb300 import api, build
    build.build()
    chs = [W.Channel(0, 0, 0, 0, 0), W.Channel(1, 1, 0, 2, 1)]
    S, nE = 5, 9
    wl = W.Workload("nan", chs, [n_wp] * 2, W.GEN_YUKAWA, W.YUKAWA_PARAMS.copy(), W.N_TERMS_YUKAWA,
                    W.coefficient_samples(S, 1), np.linspace(2.0, 300.0, nE))
    c = api.Context(0)
    md = api.Model(c, wl)
    t0, d0, s0 = gpu_run(c, md, wl)
    cf = wl.coeffs.copy()
    cf[2, 3] = bad
    t = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda:0")  # noqa: E731
    tt = torch.zeros((S, 2, nE, 2, 2, 2), dtype=torch.float64, device="cuda:0")
    d = torch.zeros((S, 2, nE, 3), dtype=torch.float64, device="cuda:0")
    sg = torch.zeros((S, nE), dtype=torch.float64, device="cuda:0")
    c.solve(md.vset, t(cf), S, t(wl.e_lab), tt, d, sg)
    assert c.sync_status() == -4
    tt, d, sg = tt.cpu().numpy(), d.cpu().numpy(), sg.cpu().numpy()
    c.close()
    keep = [0, 1, 3, 4]
    t1 = tt.view(np.complex128).reshape(S, 2, nE, 2, 2)
    assert np.array_equal(t1[keep], t0[keep]) and np.array_equal(d[keep], d0[keep]) and np.array_equal(sg[keep], s0[keep])
    assert np.isnan(tt[2, 0, :, 0, 0]).all() and np.isnan(tt[2, 1]).all() and np.isnan(sg[2]).all()
