"""Spin observables at more angles in one call than a grid has rows (65535 blocks of
32 angles): every point as in a call of its own."""
import numpy as np
import pytest

from paper_2106_00454_gb300 import inputs as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_th", [65535 * 32 + 1, 2_200_000])
def test_many_angles(n_th):
    import torch
    from paper_2106_00454_gb300 import api, build
    build.build()
    c = api.Context(0)
    chs = W.np_channels(1)
    rng = np.random.default_rng(3)
    t = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda:0")  # noqa: E731
    d, e = t(rng.uniform(-60.0, 60.0, (1, len(chs), 1, 3))), t(np.array([120.0]))
    th = t(np.linspace(0.01, np.pi - 0.01, n_th))

    def run(theta):
        a = torch.zeros((1, 1, theta.numel(), 5, 2), dtype=torch.float64, device="cuda:0")
        s = torch.zeros((1, 1, theta.numel()), dtype=torch.float64, device="cuda:0")
        c.saclay(chs, d, 1, e, theta, a, s)
        c.sync()
        return a, s

    a, s = run(th)
    for lo, hi in ((0, 70), (n_th // 2 // 32 * 32, n_th // 2 // 32 * 32 + 64), ((n_th - 1) // 32 * 32, n_th)):
        pa, ps = run(th[lo:hi].clone())
        assert torch.equal(a[:, :, lo:hi], pa) and torch.equal(s[:, :, lo:hi], ps)
    c.close()
