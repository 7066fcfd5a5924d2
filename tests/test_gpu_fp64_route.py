"""Which FP64 solves the refinement finishes: every one of the potentials that the
path is for, and none of the values that FP32 cannot hold.  (The results alone do
not tell: the FP64 Jacobi kernel gives the same ones, up to seventy times slower.)"""
import numpy as np
import pytest

from paper_2106_00454_gb300 import inputs as W

from parity_util import gpu_run
from test_gpu_fp64_refine import _fine

pytestmark = pytest.mark.gpu
UNC, CPL = W.Channel(0, 0, 0, 0, 0), W.Channel(1, 2, 1, 3, 1)


@pytest.fixture()
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_00454_gb300 import api, build
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _solve_fine(ctx, kind, ch, N, S=3):
    import torch
    n, rng = ch.K * N, np.random.default_rng(N + 7)
    v = np.stack([_fine(kind, n, N, rng), _fine(kind, n, N, rng)])
    vf = torch.tensor(v, dtype=torch.float64, device="cuda:0").contiguous()
    mid = ctx.mesh(N, n_quad=1)
    vset = ctx.project([mid], [ch], W.GEN_FINE, None, 2, v_fine=vf)
    cf = torch.tensor([[0.3], [-0.7], [0.01]], dtype=torch.float64, device="cuda:0")
    ctx.release(ctx.diag(vset, cf, S))
    ctx.sync()
    return S


@pytest.mark.parametrize("ch,N", [(UNC, 33), (UNC, 64), (UNC, 129), (CPL, 50), (CPL, 115), (CPL, 153)],
                         ids=lambda x: x if isinstance(x, int) else x.name)
def test_generic_matrices_are_refined(ctx, ch, N):
    _solve_fine(ctx, "generic", ch, N)
    assert ctx.fp64_unrefined() == 0


@pytest.mark.parametrize("exec_mode", [0, 1], ids=["batched", "plain"])
@pytest.mark.parametrize("N,S", [(32, 40), (100, 6), (150, 2)])
def test_projected_channels_are_refined(ctx, exec_mode, N, S):
    from paper_2106_00454_gb300 import api
    ctx.set_exec(exec_mode)
    chs = W.np_channels(4)
    wl = W.Workload("route", chs, [N] * len(chs), W.GEN_YUKAWA, W.YUKAWA_PARAMS.copy(), W.N_TERMS_YUKAWA,
                    W.coefficient_samples(S, 9), np.linspace(2.0, 300.0, 5))
    gpu_run(ctx, api.Model(ctx, wl), wl)
    assert ctx.fp64_unrefined() == 0


@pytest.mark.parametrize("ch,N", [(UNC, 33), (CPL, 116)], ids=lambda x: x if isinstance(x, int) else x.name)
def test_values_outside_fp32_take_fp64_jacobi(ctx, ch, N):
    assert _solve_fine(ctx, "huge", ch, N) == ctx.fp64_unrefined()
