"""FP64 solves of small matrices: the FP64 Jacobi kernel alone up to n = 16, the
refinement from n = 17 on.  Eigenpairs against LAPACK on both sides of the line
(20 n u, as for the larger sizes), few launches below it, and the same bits alone, in
a batch and with the size buckets side by side or one after another."""
import dataclasses

import numpy as np
import pytest

from paper_2106_00454_gb300 import inputs as W

from parity_util import gpu_run
from test_gpu_fp64_refine import _fine

pytestmark = pytest.mark.gpu
UNC, CPL = W.Channel(0, 0, 0, 0, 0), W.Channel(1, 1, 0, 2, 1)


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_00454_gb300 import api, build
    build.build()
    c = api.Context(0)
    yield c
    c.close()


def _wl(channels, nwp, S, n_e=5):
    return W.Workload("small", channels, nwp, W.GEN_YUKAWA, W.YUKAWA_PARAMS.copy(), W.N_TERMS_YUKAWA,
                      W.coefficient_samples(S, 11), np.linspace(2.0, 300.0, n_e))


@pytest.mark.parametrize("ch,N", [(UNC, 4), (UNC, 15), (UNC, 16), (UNC, 17), (CPL, 8), (CPL, 9)],
                         ids=lambda x: x if isinstance(x, int) else x.name)
def test_eigenpairs(ctx, orc, ch, N):
    import torch
    n, rng = ch.K * N, np.random.default_rng(N)
    v = np.stack([_fine("generic", n, N, rng) for _ in range(2)])
    mid = ctx.mesh(N, n_quad=1)
    vset = ctx.project([mid], [ch], W.GEN_FINE, None, 2,
                       v_fine=torch.tensor(v, dtype=torch.float64, device="cuda:0").contiguous())
    ctx.sync()
    V = ctx.vset_get(vset, 0)
    kb, _, _ = ctx.mesh_get(mid, N, 1)
    h0 = np.array([orc.h0(0, kb[i], kb[i + 1]) for i in range(N)])
    c = np.array([0.3, -0.7, 0.01])
    eid = ctx.diag(vset, torch.tensor(c[:, None], dtype=torch.float64, device="cuda:0"), 3)
    ctx.sync()
    u = np.finfo(float).eps
    for s in range(3):
        H = V[0] + c[s] * V[1] + np.diag(np.tile(h0, ch.K))
        eps, C = ctx.eig_get(eid, s, 0, n)
        nh = np.linalg.norm(H)
        assert np.max(np.abs(eps - np.linalg.eigvalsh(H))) <= 20 * n * u * nh
        assert np.linalg.norm(H @ C - C * eps) <= 20 * n * u * nh
        assert np.linalg.norm(C.T @ C - np.eye(n)) <= 20 * n * u
    for h in (eid, vset, mid):
        ctx.release(h)


@pytest.mark.parametrize("ch,N", [(UNC, 4), (UNC, 16), (CPL, 8)], ids=lambda x: x if isinstance(x, int) else x.name)
def test_small_solves_take_few_launches(ctx, ch, N):
    """Sum, eigensolve, plan, T and its gather and observables: one launch each, also on a
    set's first solve after the CTA size is known."""
    wl = _wl([ch], [N], 3)
    from paper_2106_00454_gb300 import api
    gpu_run(ctx, api.Model(ctx, wl), wl)  # the autotuner's calls
    md = api.Model(ctx, wl)
    k0 = ctx.kernel_launches()
    gpu_run(ctx, md, wl)
    assert ctx.kernel_launches() - k0 <= 8


def test_same_bits_alone_in_a_batch_and_on_streams(ctx):
    from paper_2106_00454_gb300 import api
    chs = [UNC, CPL, W.Channel(1, 1, 1, 1, 0), W.Channel(1, 2, 1, 3, 1), W.Channel(1, 0, 1, 1, 0)]
    wl = _wl(chs, [16, 8, 12, 9, 24], 60)
    md = api.Model(ctx, wl)
    whole = [gpu_run(ctx, md, wl) for _ in range(3)][-1]
    ctx.profile(True)  # one bucket after another
    try:
        runs = [(0, 60, gpu_run(ctx, md, wl))]
    finally:
        ctx.profile(False)
    for s, k in ((7, 1), (20, 11)):
        runs.append((s, k, gpu_run(ctx, md, dataclasses.replace(wl, coeffs=wl.coeffs[s:s + k]))))
    for s, k, r in runs:
        for x, y in zip(r, whole):
            assert np.array_equal(x, y[s:s + k])
