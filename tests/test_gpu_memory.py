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


def _wl(nwp, S, n_e=8, jmax=2):
    chs = W.np_channels(jmax)
    return W.Workload("memory", chs, [nwp[k % len(nwp)] for k in range(len(chs))], W.GEN_YUKAWA, W.YUKAWA_PARAMS.copy(),
                      W.N_TERMS_YUKAWA, W.coefficient_samples(S, 2), np.linspace(2.0, 300.0, n_e))


def _phases(ctx, md, wl, prec, n=3):
    """Solved n times: one by one, captured, replayed."""
    import torch
    S, nE = wl.n_samples, len(wl.e_lab)
    cf = torch.tensor(wl.coeffs, dtype=torch.float64, device="cuda:0")
    e = torch.tensor(wl.e_lab, dtype=torch.float64, device="cuda:0")
    d = torch.zeros((S, len(wl.channels), nE, 3), dtype=torch.float64, device="cuda:0")
    for _ in range(n):
        ctx.solve(md.vset, cf, S, e, None, d, None, prec=prec)
        ctx.sync()
    return d.cpu().numpy()


def _close(a, b, tol):
    assert np.max(np.abs(dphase(a[..., :2], b[..., :2]))) <= tol
    assert np.max(np.abs(a[..., 2] - b[..., 2])) <= tol


def _model_bytes(api, wl):
    c = api.Context(0)
    api.Model(c, wl)
    c.sync()
    n = c.bytes_in_use()
    c.close()
    return n


def test_fp64_scratch_yields_to_a_second_set(api):
    """A budget of two sets and one batch's eigenpairs and T: the refinement of the
    first set's solves takes what is there, and the second set still finds its room."""
    wl = _wl([64], 16)
    n2 = sum((ch.K * 64) ** 2 for ch in wl.channels)
    budget = 2 * _model_bytes(api, wl) + 8 * 16 * n2 + 3 * MB
    free = api.Context(0)
    want = _phases(free, api.Model(free, wl), wl, api.PREC_FP64)
    free.close()
    c = api.Context(0, hbm_budget_bytes=budget)
    first = api.Model(c, wl)
    a = _phases(c, first, wl, api.PREC_FP64)
    second = api.Model(c, wl)
    b = _phases(c, second, wl, api.PREC_FP64)
    again = _phases(c, first, wl, api.PREC_FP64)
    assert c.bytes_in_use() <= budget
    c.close()
    for x in (a, b, again):
        _close(x, want, 1e-8)


def test_shares_of_the_streams_yield_to_a_second_set(api):
    """Mixed path, a budget of one size bucket's scratch at a time and a second set: the
    shares for buckets side by side (5 MB more) may take the second set's room (7 MB), but
    not keep it."""
    wl = _wl([64], 2)
    probe = api.Context(0)
    probe.profile(True)  # one bucket after another
    md = api.Model(probe, wl)
    want = _phases(probe, md, wl, api.PREC_MIXED)
    one = probe.bytes_in_use()
    probe.close()
    budget = one + _model_bytes(api, wl) + MB // 16
    c = api.Context(0, hbm_budget_bytes=budget)
    first = api.Model(c, wl)
    a = _phases(c, first, wl, api.PREC_MIXED, 4)
    api.Model(c, wl)
    b = _phases(c, first, wl, api.PREC_MIXED)
    assert c.bytes_in_use() <= budget
    c.close()
    assert np.array_equal(a, want) and np.array_equal(b, want)


def test_served_fp64_under_a_budget(api):
    """The scratch of a served FP64 batch is no part of what admission counts, yields to a
    set that the program projects meanwhile, and the synchronous calls' scratch yields to
    the server's batches."""
    chs = W.np_channels(2)
    rng = np.random.default_rng(8)
    req = {n: (rng.standard_normal(14) * W.TERM_SCALE, np.sort(rng.uniform(1.0, 350.0, 20)), n) for n in (64, 96)}
    args = (chs, W.GEN_YUKAWA, W.YUKAWA_PARAMS, W.N_TERMS_YUKAWA, [64, 96])

    def ask(c, n):
        r = c.wait(c.submit(*req[n], api.PREC_FP64))
        assert r.status == 0
        return r.delta

    probe = api.Context(0)
    probe.serve_start(*args, max_batch=4, n_slots=1)
    want = {n: ask(probe, n) for n in (64, 96)}
    probe.serve_stop()
    probe.close()
    probe = api.Context(0)
    probe.serve_start(*args, max_batch=4, n_slots=1)
    base = probe.bytes_in_use()
    probe.serve_stop()
    probe.close()
    wl = _wl([64], 4)
    need96 = 8 * sum((ch.K * 96) ** 2 for ch in chs)
    # the server, a further set, and room for one request's eigenpairs and T (and little more)
    budget = base + _model_bytes(api, wl) + need96 + 8 * 4 * sum((ch.K * 64) ** 2 for ch in chs) + MB
    c = api.Context(0, hbm_budget_bytes=budget)
    c.serve_start(*args, max_batch=4, n_slots=1)
    try:
        for _ in range(3):  # the first batch's scratch takes what is left
            _close(ask(c, 64), want[64], 1e-8)
        md = api.Model(c, wl)
        _close(ask(c, 64), want[64], 1e-8)
        _phases(c, md, wl, api.PREC_FP64)
        _close(ask(c, 96), want[96], 1e-8)  # more eigenpairs than the slot holds
        _close(ask(c, 64), want[64], 1e-8)
        assert c.bytes_in_use() <= budget
    finally:
        c.serve_stop()
        c.close()


def test_streams_are_taken_up_again_when_room_returns(api):
    """Mixed path, two sets and one bucket's scratch at a time: no shares for the streams
    (5 MB more); once the second set (7 MB) is released the next solves take them."""
    wl = _wl([64], 2)
    probe = api.Context(0)
    probe.profile(True)  # one bucket after another
    first = api.Model(probe, wl)
    api.Model(probe, wl)
    want = _phases(probe, first, wl, api.PREC_MIXED)
    budget = probe.bytes_in_use() + MB
    probe.close()
    c = api.Context(0, hbm_budget_bytes=budget)
    first, second = api.Model(c, wl), api.Model(c, wl)
    a = _phases(c, first, wl, api.PREC_MIXED, 4)
    second.release()
    before = c.bytes_in_use()
    b = _phases(c, first, wl, api.PREC_MIXED)
    assert before + 4 * MB < c.bytes_in_use() <= budget
    c.close()
    assert np.array_equal(a, want) and np.array_equal(b, want)


def test_server_and_program_share_a_tight_budget(api):
    """A program projects, solves and releases while the server works through FP64 and
    mixed requests, under a budget in which each needs the other's spare scratch: every
    call finishes, with the results that it has alone."""
    import threading
    chs = W.np_channels(2)
    rng = np.random.default_rng(12)
    reqs = [(rng.standard_normal(14) * W.TERM_SCALE, np.sort(rng.uniform(1.0, 350.0, 12)), (48, 64)[k % 2], k // 2 % 2)
            for k in range(12)]
    args = (chs, W.GEN_YUKAWA, W.YUKAWA_PARAMS, W.N_TERMS_YUKAWA, [48, 64])
    wl = _wl([64], 6)
    free = api.Context(0)
    want_p = _phases(free, api.Model(free, wl), wl, api.PREC_FP64)
    free.serve_start(*args, max_batch=2, n_slots=2)
    want_r = [free.wait(free.submit(*r)).delta for r in reqs]
    held = free.bytes_in_use()
    free.close()
    # what the server and the program need to keep, the mixed slots' scratch, a second set, and a little
    c = api.Context(0, hbm_budget_bytes=held + _model_bytes(api, wl) - 44 * MB)
    c.serve_start(*args, max_batch=2, n_slots=2)
    bad = []

    def serve():
        try:
            for k in range(60):
                r = c.wait(c.submit(*reqs[k % len(reqs)]))
                assert r.status == 0, r.status
                _close(r.delta, want_r[k % len(reqs)], 1e-3 if reqs[k % len(reqs)][3] else 1e-8)
        except Exception as ex:  # noqa: BLE001
            bad.append(repr(ex))

    th = threading.Thread(target=serve)
    th.start()
    try:
        for _ in range(15):
            md = api.Model(c, wl)
            _close(_phases(c, md, wl, api.PREC_FP64, 2), want_p, 1e-8)
            md.release()
    finally:
        th.join(120)
    assert not th.is_alive() and not bad, bad
    c.serve_stop()
    c.close()
