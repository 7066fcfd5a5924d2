"""FP64 eigenpairs through the FP32 solve and the tensor-core refinement, and
the FP64 Jacobi kernel that takes what the refinement does not.

Eigenpairs of caller-supplied potentials against numpy at the sizes where the
path changes: odd and tiny matrices, the digit products' tile and chunk edges
(64, 128, 32), the FP64 and FP32 shared-memory limits, one size above both.
Potentials: a generic one; none at all and a weak coupling of the two l-blocks
(the coupled H0 is doubly degenerate, so the eigenvalue pairs lie anywhere from
equal to barely resolved); and one too large for FP32, which has to come out of
the FP64 Jacobi kernel.  Bounds: 20 n u in the residual and the orthogonality,
relative to ||H||_F (the backward error of an FP64 eigensolve, n sweeps' worth
of rounding), as for the eigenpair test of the projected channels."""
import numpy as np
import pytest

from paper_2106_00454_gb300 import inputs as W

pytestmark = pytest.mark.gpu


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


def _fine(kind, n, N, rng):
    """Symmetric fine-grid values (one point per bin) of one term."""
    if kind == "none":
        return np.zeros((n, n))
    B = rng.standard_normal((n, n))
    v = 0.02 * (B + B.T)
    if kind == "weak":  # l-blocks coupled a little, each block untouched
        v *= 10.0 ** rng.uniform(-14.0, -4.0, (n, 1))
        v = v + v.T
        v[:N, :N] = 0.0
        v[N:, N:] = 0.0
    if kind == "huge":
        v *= 1e42
    return v


CASES = [("generic", 0, N) for N in (4, 5, 31, 33, 64, 65, 128, 129)] + \
        [("generic", 1, N) for N in (4, 33, 50, 115, 116, 152, 153)] + \
        [("none", 1, N) for N in (7, 64)] + [("weak", 1, N) for N in (9, 64, 100)] + \
        [("huge", 0, 24), ("huge", 1, 116)]


@pytest.mark.parametrize("kind,coupled,N", CASES, ids=[f"{k}-{'c' if c else 'u'}{N}" for k, c, N in CASES])
def test_eigenpairs(ctx, orc, kind, coupled, N):
    import torch
    ch = W.Channel(1, 2, 1, 3, 1) if coupled else W.Channel(0, 0, 0, 0, 0)
    n, rng = ch.K * N, np.random.default_rng(N + 1000 * coupled)
    S = 3
    v = np.stack([_fine(kind, n, N, rng), _fine("none" if kind in ("none", "weak") else kind, n, N, rng)])
    vf = torch.tensor(v, dtype=torch.float64, device="cuda:0").contiguous()
    mid = ctx.mesh(N, n_quad=1)
    vset = ctx.project([mid], [ch], W.GEN_FINE, None, 2, v_fine=vf)
    ctx.sync()
    V = ctx.vset_get(vset, 0)
    kb, _, _ = ctx.mesh_get(mid, N, 1)
    h0 = np.array([orc.h0(0, kb[i], kb[i + 1]) for i in range(N)])
    c = np.array([0.3, -0.7, 0.01])
    cf = torch.tensor(c[:, None], dtype=torch.float64, device="cuda:0")
    eid = ctx.diag(vset, cf, S)
    st = torch.zeros((S, 1), dtype=torch.int32, device="cuda:0")
    ctx.diag_status(eid, st)
    ctx.sync()
    assert (st.cpu().numpy() > 0).all() or kind == "none"
    u = np.finfo(float).eps
    for s in range(S):
        H = V[0] + c[s] * V[1] + np.diag(np.tile(h0, ch.K))
        eps, C = ctx.eig_get(eid, s, 0, n)
        nh = np.linalg.norm(H)
        assert np.all(np.diff(eps) >= 0)
        assert np.max(np.abs(eps - np.linalg.eigvalsh(H))) <= 20 * n * u * nh
        assert np.linalg.norm(H @ C - C * eps) <= 20 * n * u * nh
        assert np.linalg.norm(C.T @ C - np.eye(n)) <= 20 * n * u
    for h in (eid, vset, mid):
        ctx.release(h)


def test_budget_without_room_for_the_refinement(ctx):
    """A context whose budget leaves no room for the refinement's scratch still
    solves (FP64 Jacobi alone), to the same phases."""
    import torch
    from paper_2106_00454_gb300 import api
    wl = W.workload_all_channels(n_wp=40, jmax=1, n_e=16)

    def phases(c):
        md = api.Model(c, wl)
        cf = torch.tensor(wl.coeffs, dtype=torch.float64, device="cuda:0")
        e = torch.tensor(wl.e_lab, dtype=torch.float64, device="cuda:0")
        d = torch.zeros((1, len(wl.channels), 16, 3), dtype=torch.float64, device="cuda:0")
        for _ in range(3):  # one by one, captured, replayed
            c.solve(md.vset, cf, 1, e, None, d, None)
            c.sync()
        return d.cpu().numpy(), c.bytes_in_use()

    probe = api.Context(0)
    probe.set_exec(api.EXEC_PLAIN)
    md = api.Model(probe, wl)
    room = probe.bytes_in_use() + (3 << 20)
    probe.close()
    tight = api.Context(0, hbm_budget_bytes=room)
    a, used = phases(tight)
    tight.close()
    b, _ = phases(ctx)
    assert used <= room
    assert np.max(np.abs((a - b + 90.0) % 180.0 - 90.0)) <= 1e-8
