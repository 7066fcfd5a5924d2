"""FP64 eigenpairs of projected channels at the refinement's own bounds, up to the
largest matrices: the stopping test leaves at most 2e-14 of ||H||_F, the 55-bit
products and the rounding of X n u per Frobenius norm and factor (four of them in
X^T X and H X); eigenvalues 2e-14 plus LAPACK's few u.  The refinement finishes all
of them, and T above n = 512 agrees with the oracle at the FP64 tolerances."""
import numpy as np
import pytest

from paper_2106_00454_gb300 import inputs as W

from parity_util import compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu
UNC, CPL = W.Channel(0, 0, 0, 0, 0), W.Channel(1, 1, 0, 2, 1)


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_00454_gb300 import api, build
    build.build()
    return api


@pytest.mark.parametrize("ch,N", [(UNC, 17), (UNC, 64), (CPL, 64), (UNC, 150), (CPL, 150), (CPL, 256), (CPL, 257), (CPL, 512)],
                         ids=lambda x: x if isinstance(x, int) else x.name)
def test_eigenpairs_at_the_stopping_bound(api, orc, ch, N):
    import torch
    ctx = api.Context(0)
    S, n = 3, ch.K * N
    wl = W.Workload("bounds", [ch], [N], W.GEN_YUKAWA, W.YUKAWA_PARAMS.copy(), W.N_TERMS_YUKAWA,
                    W.coefficient_samples(S, 13), np.linspace(2.0, 300.0, 3))
    md = api.Model(ctx, wl)
    V = ctx.vset_get(md.vset, 0)
    kb, _, _ = ctx.mesh_get(md.mesh_of_n[N], N, W.MESH_Q)
    h0 = np.array([orc.h0(0, kb[i], kb[i + 1]) for i in range(N)])
    eid = ctx.diag(md.vset, torch.tensor(wl.coeffs, dtype=torch.float64, device="cuda:0"), S)
    ctx.sync()
    u = np.finfo(float).eps
    for s in range(S):
        H = V[0] + np.tensordot(wl.coeffs[s], V[1:], 1) + np.diag(np.tile(h0, ch.K))
        eps, C = ctx.eig_get(eid, s, 0, n)
        nh = np.linalg.norm(H)
        assert np.max(np.abs(eps - np.linalg.eigvalsh(H))) <= (2e-14 + 20 * u) * nh
        assert np.linalg.norm(H @ C - C * eps) <= (2e-14 + 4 * n * u) * nh
        assert np.linalg.norm(C.T @ C - np.eye(n)) <= 2e-14 + 4 * n * u
    assert ctx.fp64_unrefined() == 0
    ctx.close()


def test_t_above_n_512_matches_the_oracle(api, orc):
    ctx = api.Context(0)
    wl = W.Workload("large", [CPL], [260], W.GEN_YUKAWA, W.YUKAWA_PARAMS.copy(), W.N_TERMS_YUKAWA,
                    W.coefficient_samples(1, 17), np.linspace(2.0, 300.0, 7))
    compare(wl, gpu_run(ctx, api.Model(ctx, wl), wl), oracle_run(orc, wl))
    ctx.close()


@pytest.mark.parametrize("ch,N", [(UNC, 33), (UNC, 65), (UNC, 129)], ids=lambda x: x if isinstance(x, int) else x.name)
def test_update_shared_by_two_four_and_eight_ctas_same_bits(api, ch, N):
    """The refinement's update takes clusters of up to 8 CTAs, two rows a warp of 8 or more
    (n >= 16 a CTA) and two CTAs an SM: 2, 4 and 8 of them a matrix, against one."""
    import dataclasses
    ctx = api.Context(0)
    wl = W.Workload("shares", [ch], [N], W.GEN_YUKAWA, W.YUKAWA_PARAMS.copy(), W.N_TERMS_YUKAWA,
                    W.coefficient_samples(400, 19), np.linspace(2.0, 300.0, 3))
    md = api.Model(ctx, wl)
    whole = gpu_run(ctx, md, wl)
    for s, k in ((3, 2), (40, 60), (200, 140)):
        part = gpu_run(ctx, md, dataclasses.replace(wl, coeffs=wl.coeffs[s:s + k]))
        for x, y in zip(part, whole):
            assert np.array_equal(x, y[s:s + k])
    ctx.close()
