"""Calls with little device memory: what a call can do without (the forms of the
solvers that are only faster) yields to what any call needs."""
import numpy as np
import pytest

from paper_2106_00454_gb300 import inputs as W

from parity_util import dphase

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_00454_gb300 import api, build
    build.build()
    return api


class Inversion:
    """An inversion with enough systems for the eigendecompositions."""

    def __init__(self, nq, S, n_I, jmax=4):
        import torch
        self.nq, self.S, self.chs = nq, S, W.np_channels(jmax)
        t = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda:0")  # noqa: E731
        self.cf, self.ei, self.el = t(W.coefficient_samples(S, 4)), t(W.chebyshev_energies(n_I)), t(W.lab_energies(7))
        self.d = torch.zeros((S, len(self.chs), 7, 3), dtype=torch.float64, device="cuda:0")
        assert S * len(self.chs) * n_I >= 12 * 152

    def prepare(self, ctx):
        return ctx.mi_prepare(self.chs, W.GEN_YUKAWA, W.YUKAWA_PARAMS, W.N_TERMS_YUKAWA, n_quad=self.nq)

    def solve(self, ctx, mid):
        self.d.zero_()
        ctx.mi_solve(mid, self.cf, self.S, self.ei, self.el, None, self.d, None)
        ctx.sync()
        return self.d.cpu().numpy()

    def same(self, a, b):
        assert np.max(np.abs(dphase(a[..., :2], b[..., :2]))) <= 1e-8


def test_inversion_under_a_budget_of_its_inputs_and_elimination(api):
    """The terms, the on-shell rows, the phases and one slot of two matrices per
    (sample, channel): what the elimination alone needs."""
    iv = Inversion(24, 64, 16)
    M, Ks = iv.nq + 1, np.array([ch.K for ch in iv.chs])
    inputs = 8 * W.N_TERMS_YUKAWA * int(np.sum((Ks * M) ** 2))
    onshell = 8 * 16 * W.N_TERMS_YUKAWA * int(np.sum(Ks ** 2)) * M
    phases = 8 * iv.S * len(Ks) * 16 * 3 + 4 * iv.S * len(Ks)
    slots = max(2 * 8 * (K * M) ** 2 * iv.S * int(np.sum(Ks == K)) for K in (1, 2))
    budget = inputs + onshell + phases + slots + MB // 4
    free = api.Context(0)
    want = iv.solve(free, iv.prepare(free))
    free.close()
    tight = api.Context(0, hbm_budget_bytes=budget)
    got = iv.solve(tight, iv.prepare(tight))
    assert tight.bytes_in_use() <= budget
    tight.close()
    iv.same(got, want)


def test_inversion_on_a_nearly_full_device(api):
    """Room for the eigenpairs or for the elimination's slots (92 MB), not for both."""
    import torch
    iv = Inversion(96, 64, 32)
    eig = 8 * iv.S * sum((ch.K * iv.nq) ** 2 for ch in iv.chs)
    ctx = api.Context(0)
    want = iv.solve(ctx, iv.prepare(ctx))  # also loads every kernel
    ctx.close()
    ctx = api.Context(0)
    mid = iv.prepare(ctx)
    ctx.sync()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - eig - 34 * MB, dtype=torch.uint8, device="cuda:0")
    try:
        got = iv.solve(ctx, mid)
    finally:
        del fill
        torch.cuda.empty_cache()
        ctx.close()
    iv.same(got, want)
