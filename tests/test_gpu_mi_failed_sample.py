"""An inversion of many systems (one eigendecomposition per sample and channel) with a
sample that has no solution: its eigensolves fail and are left to elimination, which
says what it says of the sample alone; the other samples keep their bits."""
import numpy as np
import pytest

from paper_2106_00454_gb300 import inputs as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("nq,S,n_I", [(8, 60, 17), (33, 41, 14)])
def test_failed_sample_is_left_to_elimination(nq, S, n_I, bad):
    import torch
    from paper_2106_00454_gb300 import api, build
    build.build()
    chs = W.np_channels(2)
    assert S * len(chs) * n_I >= 12 * 152
    c = api.Context(0)
    mid = c.mi_prepare(chs, W.GEN_YUKAWA, W.YUKAWA_PARAMS, W.N_TERMS_YUKAWA, n_quad=nq)
    t = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda:0")  # noqa: E731
    ei, el = t(W.chebyshev_energies(n_I)), t(W.lab_energies(5))

    def run(cf):
        n = len(cf)
        d = torch.zeros((n, len(chs), 5, 3), dtype=torch.float64, device="cuda:0")
        st = torch.full((n, len(chs)), 99, dtype=torch.int32, device="cuda:0")
        c.mi_solve(mid, t(cf), n, ei, el, None, d, None, st)
        return c.sync_status(), d.cpu().numpy(), st.cpu().numpy()

    cf = W.coefficient_samples(S, 6)
    for _ in range(2):  # the second call runs both block sizes side by side
        rc, d0, s0 = run(cf)
        assert rc == 0 and (s0 > 0).all()
    cf = cf.copy()
    cf[7, 0] = bad
    rc, d1, s1 = run(cf)
    rc_alone, d_alone, s_alone = run(cf[7:8])  # few systems: by elimination
    keep = np.arange(S) != 7
    assert rc == rc_alone and np.array_equal(s1[7], s_alone[0])
    assert np.isnan(d1[7][:, :, 0]).all() and np.isnan(d_alone[0][:, :, 0]).all()
    assert np.array_equal(d1[keep], d0[keep]) and np.array_equal(s1[keep], s0[keep])
    c.close()
