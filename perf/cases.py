"""Performance cases: what a user of this library has it do, through its public entry points.

Each case is one call (or one burst of served requests) of the kinds that a study of
nucleon-nucleon scattering makes: a single phase-shift curve, all partial waves of one
parameter set, ensembles of parameter samples in FP64 and in mixed precision, large
wave-packet bases, the point resolvent, the matrix-inversion method, spin observables,
and a burst of requests to the server.

``listed()`` names them, ``draw`` gives more of the same ranges, ``prepare`` makes the
inputs from a seed, ``run`` makes the call, ``work`` says what it cannot do without, and
``exact`` is the same result in plain 64-bit torch.
"""
import concurrent.futures
import math

import numpy as np
import torch

from paper_2106_00454_gb300 import api
from paper_2106_00454_gb300 import inputs as W

DEV = "cuda:0"
F64 = torch.float64


# ------------------------------------------------------------------------------------ cases
def _case(name, kind, **kw):
    c = {
        "kind": kind,            # solve | host | mi | spin | serve
        "pot": "yukawa",         # yukawa | yamaguchi
        "jmax": 4,               # partial waves up to this J (-1: 1S0 alone)
        "tz_copy": True,         # the T_z = +-1 copy of 1S0 beside the np channels
        "n_wp": "64",            # N_WP, or the sizes from which each channel draws its own
        "wp_kind": W.WP_MOMENTUM,
        "samples": 1,
        "energies": 128,
        "even": True,            # energies evenly spaced over 1..350 MeV, else drawn from the seed
        "prec": api.PREC_FP64,
        "proj": api.PREC_FP64,
        "res": api.AVG_FREE_BIN,
        "n_int": 0,              # mi: interpolation energies
        "n_quad": 0,             # mi: grid points
        "angles": 0,             # spin: scattering angles
    }
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one phase-shift curve of a model potential: the smallest call, bound by launches and latency
        _case("curve_1s0_fp64", "solve", pot="yamaguchi", jmax=-1, tz_copy=False, n_wp="32", energies=64, even=False),
        # every partial wave of one parameter set, as in a cross-section prediction
        _case("all_waves_fp64", "solve", jmax=6, tz_copy=False, n_wp="100", energies=100),
        # a small posterior ensemble in full precision, N_WP chosen per channel
        _case("ensemble_fp64", "solve", n_wp="40,64,100", samples=256),
        # converged reference results in the largest FP64 basis of the ensemble studies (coupled 300 x 300)
        _case("reference_150_fp64", "solve", jmax=6, tz_copy=False, n_wp="150", samples=8),
        # odd sizes, energy packets and the resolvent without averaging
        _case("point_odd_fp64", "solve", jmax=3, tz_copy=False, n_wp="51", wp_kind=W.WP_ENERGY, samples=33, energies=61,
              even=False, res=api.POINT),
        # a parameter set asked for on the host, as a fit's objective function does
        _case("one_set_host_mixed", "host", n_wp="64", energies=37, even=False, prec=api.PREC_MIXED),
        # ensembles in mixed precision: the mixed-size channel set ...
        _case("ensemble_mixed", "solve", n_wp="40,64,100", samples=1024, prec=api.PREC_MIXED),
        # ... and the large basis with the reduced-precision projection: the library's headline workload
        _case("posterior_150_mixed", "solve", jmax=6, tz_copy=False, n_wp="150", samples=1024, prec=api.PREC_MIXED,
              proj=api.PREC_MIXED),
        # the largest served basis (coupled 512 x 512)
        _case("large_256_mixed", "solve", n_wp="256", samples=16, energies=93, prec=api.PREC_MIXED),
        # the comparison method at Chebyshev energies
        _case("inversion_ensemble", "mi", samples=64, n_int=32, n_quad=96),
        # spin amplitudes and differential cross sections over an ensemble's phase shifts
        _case("spin_ensemble", "spin", tz_copy=False, samples=256, angles=32),
        # a burst of requests with their own energies and sizes
        _case("served_burst_mixed", "serve", n_wp="32,64", samples=48, prec=api.PREC_MIXED),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "solve", "host", "mi", "spin", "serve"])
    if kind == "mi":
        return _case(None, "mi", jmax=rng.randint(0, 4), tz_copy=rng.random() < 0.5, samples=_log_int(rng, 1, 64),
                     n_int=rng.randint(8, 32), n_quad=rng.randint(24, 96), energies=_log_int(rng, 16, 256))
    if kind == "spin":
        return _case(None, "spin", jmax=rng.randint(1, 6), tz_copy=False, samples=_log_int(rng, 1, 256),
                     energies=_log_int(rng, 8, 128), angles=rng.randint(1, 32))
    prec = rng.choice([api.PREC_FP64, api.PREC_MIXED])
    if kind == "serve":
        sizes = rng.choice(["32", "48,64", "37,64", "32,64"])
        return _case(None, "serve", jmax=rng.randint(1, 4), n_wp=sizes, samples=_log_int(rng, 4, 48),
                     energies=_log_int(rng, 16, 128), prec=prec)
    jmax = rng.randint(0, 6)
    n_wp = _log_int(rng, 20, 256 if prec == api.PREC_MIXED else 150)
    sizes = str(n_wp) if rng.random() < 0.7 else "%d,%d" % (n_wp, max(20, (2 * n_wp) // 3))
    c = _case(None, kind, jmax=jmax, tz_copy=rng.random() < 0.5, n_wp=sizes, energies=_log_int(rng, 16, 256),
              even=rng.random() < 0.5, prec=prec)
    if kind == "solve":
        c["wp_kind"] = rng.choice([W.WP_MOMENTUM, W.WP_MOMENTUM, W.WP_ENERGY])
        c["res"] = rng.choice([api.AVG_FREE_BIN, api.AVG_FREE_BIN, api.POINT])
        if prec == api.PREC_MIXED:
            c["proj"] = rng.choice([api.PREC_FP64, api.PREC_MIXED])
    # as many samples as keep the matrix work (sum of n^3) well inside the largest listed case's
    cap = 2e10 if prec == api.PREC_MIXED else 1.2e9
    unit = sum((ch.K * n) ** 3 for ch, n in zip(_channels(c), _sizes(c)))
    c["samples"] = _log_int(rng, 1, max(1, min(256 if kind == "solve" else 32, int(cap / unit))))
    return c


def _channels(c):
    if c["jmax"] < 0:
        return [W.Channel(0, 0, 0, 0, 0)]
    return W.np_channels(c["jmax"], extra_1s0_tz=c["tz_copy"])


def _sizes(c):
    """N_WP per channel: one size for all, or a fixed draw from several."""
    choices = [int(x) for x in c["n_wp"].split(",")]
    chs = _channels(c)
    if len(choices) == 1:
        return choices * len(chs)
    return [int(x) for x in np.random.default_rng(W.SEED + 1).choice(np.array(choices), size=len(chs))]


# ------------------------------------------------------------------------------------ inputs
_kept = {}  # the context and the projected models and servers that a program keeps for its lifetime


def _context():
    if "ctx" not in _kept:
        _kept["ctx"] = api.Context(0)
    return _kept["ctx"]


def _workload(c):
    yam = c["pot"] == "yamaguchi"
    terms = 1 if yam else W.N_TERMS_YUKAWA
    return W.Workload("case", _channels(c), _sizes(c), W.GEN_YAMAGUCHI if yam else W.GEN_YUKAWA,
                      W.YAMAGUCHI_PARAMS if yam else W.YUKAWA_PARAMS, terms, np.zeros((c["samples"], terms - 1)),
                      np.zeros(0), wp_kind=c["wp_kind"])


def _model(c):
    key = ("model", c["pot"], c["jmax"], c["tz_copy"], c["n_wp"], c["wp_kind"], c["proj"])
    if key not in _kept:
        _kept[key] = api.Model(_context(), _workload(c), proj_prec=c["proj"])
    return _kept[key]


def _inversion(c):
    key = ("mi", c["jmax"], c["tz_copy"], c["n_quad"])
    if key not in _kept:
        _kept[key] = _context().mi_prepare(_channels(c), W.GEN_YUKAWA, W.YUKAWA_PARAMS, W.N_TERMS_YUKAWA,
                                           n_quad=c["n_quad"])
    return _kept[key]


def _server(c):
    key = ("serve", c["jmax"], c["tz_copy"], c["n_wp"])
    if key not in _kept:
        srv = api.Context(0)  # a server has a context of its own
        srv.serve_start(_channels(c), W.GEN_YUKAWA, W.YUKAWA_PARAMS, W.N_TERMS_YUKAWA,
                        [int(x) for x in c["n_wp"].split(",")])
        _kept[key] = srv
    return _kept[key]


def _draws(c, seed):
    """Coefficients and energies of the case for a seed (host arrays)."""
    rng = np.random.default_rng(seed)
    if c["kind"] == "serve":
        shape = np.random.default_rng(W.SEED + 5)  # the burst's lengths and sizes are the case's, its values the seed's
        sizes = [int(x) for x in c["n_wp"].split(",")]
        reqs = []
        for _ in range(c["samples"]):
            n_e, n_wp = int(shape.integers(16, c["energies"] + 1)), int(shape.choice(sizes))
            reqs.append((rng.standard_normal(14) * W.TERM_SCALE, np.sort(rng.uniform(1.0, 350.0, n_e)), n_wp))
        return reqs
    if c["kind"] == "spin":
        # phase shifts that fall with energy and J, different in every sample
        chs, S, e = _channels(c), c["samples"], W.lab_energies(c["energies"])
        d = rng.uniform(-60.0, 60.0, (S, len(chs), 1, 3)) * np.exp(-rng.uniform(0.2, 2.0, (S, len(chs), 1, 3)) * e[:, None] / 350.0)
        damp = np.array([[1.0, 1.0, 0.1] if ch.coupled else [1.0, 0.0, 0.0] for ch in chs]) \
            / np.array([1.0 + ch.J for ch in chs])[:, None]
        return d * damp[None, :, None, :], e, np.sort(rng.uniform(0.01, np.pi - 0.01, c["angles"]))
    cf = None if c["pot"] == "yamaguchi" else rng.standard_normal((c["samples"], 14)) * W.TERM_SCALE
    e = W.lab_energies(c["energies"]) if c["even"] else np.sort(rng.uniform(1.0, 350.0, c["energies"]))
    return cf, e


def _out(*shape):
    return torch.empty(shape, dtype=F64, device=DEV)


def prepare(case, seed):
    c = case
    S, nE, nch = c["samples"], c["energies"], len(_channels(c))
    if c["kind"] == "serve":
        return {"kind": "serve", "ctx": _server(c), "reqs": _draws(c, seed), "prec": c["prec"]}
    ctx = _context()
    st = {"kind": c["kind"], "ctx": ctx, "S": S, "prec": c["prec"], "res": c["res"]}
    if c["kind"] == "spin":
        delta, e, th = (torch.tensor(x, dtype=F64, device=DEV) for x in _draws(c, seed))
        st.update(channels=_channels(c), delta=delta, e=e, th=th, abcde=_out(S, nE, c["angles"], 5, 2),
                  dsig=_out(S, nE, c["angles"]))
        return st
    cf, e = _draws(c, seed)
    if c["kind"] == "mi":
        st.update(mi=_inversion(c), cf=torch.tensor(cf, dtype=F64, device=DEV), e=torch.tensor(e, dtype=F64, device=DEV),
                  e_int=torch.tensor(W.chebyshev_energies(c["n_int"]), dtype=F64, device=DEV),
                  k=_out(S, nch, c["n_int"], 2, 2), d=_out(S, nch, nE, 3), s=_out(S, nE))
        return st
    st["vset"] = _model(c).vset
    if c["kind"] == "host":
        pin = lambda *shape: torch.empty(shape, dtype=F64, pin_memory=True)  # noqa: E731
        bufs = [pin(S, nch, nE, 2, 2, 2), pin(S, nch, nE, 3), pin(S, nE)]
        cfp, ep = pin(S, 14), pin(nE)
        cfp.copy_(torch.from_numpy(cf))
        ep.copy_(torch.from_numpy(e))
        st.update(hold=bufs + [cfp, ep], cf=cfp.numpy(), e=ep.numpy(), t=bufs[0].numpy(), d=bufs[1].numpy(), s=bufs[2].numpy())
        return st
    st.update(cf=None if cf is None else torch.tensor(cf, dtype=F64, device=DEV), e=torch.tensor(e, dtype=F64, device=DEV),
              t=_out(S, nch, nE, 2, 2, 2), d=_out(S, nch, nE, 3), s=_out(S, nE))
    return st


# ------------------------------------------------------------------------------------ calls
def run(state):
    st, ctx = state, state["ctx"]
    if st["kind"] == "serve":
        tickets = [ctx.submit(cf, e, n, prec=st["prec"]) for cf, e, n in st["reqs"]]
        got = []
        for t in tickets:
            got.append(ctx.wait(t))
            ctx.release_result(t)
        return {"T": np.concatenate([r.T.reshape(-1) for r in got]), "delta": np.concatenate([r.delta.reshape(-1) for r in got]),
                "sigma": np.concatenate([r.sigma for r in got]), "status": np.array([r.status for r in got])}
    if st["kind"] == "spin":
        ctx.saclay(st["channels"], st["delta"], st["S"], st["e"], st["th"], st["abcde"], st["dsig"])
        return {"abcde": st["abcde"], "dsig": st["dsig"]}
    if st["kind"] == "mi":
        ctx.mi_solve(st["mi"], st["cf"], st["S"], st["e_int"], st["e"], st["k"], st["d"], st["s"])
        return {"K": st["k"], "delta": st["d"], "sigma": st["s"]}
    solve = ctx.solve_host if st["kind"] == "host" else ctx.solve
    solve(st["vset"], st["cf"], st["S"], st["e"], st["t"], st["d"], st["s"], prec=st["prec"], res=st["res"])
    return {"T": st["t"], "delta": st["d"], "sigma": st["s"]}


def work(case):
    """Bytes: inputs (potential terms, coefficients, energies) and outputs once.  Operations: per channel and
    sample the paper's (8/3) n^3 of the eigendecomposition and 2 K m n^2 + 8 K^2 m n of the on-shell T at m bins
    (solves); (2/3) n^3 of one factorisation per energy (inversion); the coupling sum and the five traces (spin)."""
    c = case
    chs, S, nE = _channels(c), c["samples"], c["energies"]
    if c["kind"] == "spin":
        terms = sum(sum(1 for _ in range((2 * ch.s + 1) ** 2 * ch.K ** 2)) for ch in chs)
        pts = S * nE * c["angles"]
        return {"bytes": 8.0 * (S * len(chs) * nE * 3 + pts * 11), "flops": float(pts * (4 * terms + 400))}
    if c["kind"] == "mi":
        n = [ch.K * (c["n_quad"] + 1) for ch in chs]
        out = S * (len(chs) * (c["n_int"] * 4 + nE * 3) + nE)
        return {"bytes": 8.0 * (15 * sum(x * x for x in n) + 14 * S + out),
                "flops": float(S * c["n_int"] * sum(2.0 / 3.0 * x ** 3 for x in n))}
    sizes = _sizes(c)
    if c["kind"] == "serve":
        choices = [int(x) for x in c["n_wp"].split(",")]
        sizes = [sum(choices) / len(choices)] * len(chs)
        nE = (16 + nE) / 2
    terms = 1 if c["pot"] == "yamaguchi" else W.N_TERMS_YUKAWA
    flops = by = 0.0
    for ch, N in zip(chs, sizes):
        n, m = ch.K * N, (nE if c["res"] == api.POINT else min(N, nE + 2))
        flops += 8.0 / 3.0 * n ** 3 + 2.0 * ch.K * m * n * n + 8.0 * ch.K ** 2 * m * n
        by += terms * n * n
    return {"bytes": 8.0 * (by + (terms - 1) * S + nE + S * (len(chs) * nE * 11 + nE)), "flops": flops * S}


# ------------------------------------------------------------------------------------ the same results in plain 64 bits
HBARC, M_N = 197.3269804, 938.918309
MU = 0.5 * M_N / HBARC


def _t(x):
    return torch.as_tensor(np.asarray(x), dtype=F64, device=DEV)


def _momentum(e):
    return torch.sqrt(M_N * e / 2.0) / HBARC


def _mesh(N, wp_kind):
    th = math.atan((W.MESH_KMAX_FM / W.MESH_ALPHA_FM) ** (1.0 / W.MESH_T))
    kb = W.MESH_ALPHA_FM * np.tan(np.arange(N + 1) * th / N) ** W.MESH_T
    kb[N] = W.MESH_KMAX_FM
    x, w = np.polynomial.legendre.leggauss(W.MESH_Q)
    a, b = kb[:-1, None], kb[1:, None]
    kq, wq = (0.5 * (a + b) + 0.5 * (b - a) * x).ravel(), (0.5 * (b - a) * w).ravel()
    a, b = kb[:-1], kb[1:]
    if wp_kind == W.WP_MOMENTUM:
        norm, h0, f = b - a, (b ** 3 - a ** 3) / (3.0 * (b - a)) / (2.0 * MU), np.ones_like(kq)
    else:
        norm, h0, f = (b * b - a * a) / (2.0 * MU), 0.5 * (a * a + b * b) / (2.0 * MU), np.sqrt(kq / MU)
    return kb, kq, wq * kq * f / np.sqrt(np.repeat(norm, W.MESH_Q)), norm, h0


def _angle_integrals(pa, pb, lmax):
    """I_L[m](pa_i, pb_j) of the three Yukawa masses: [3][L][i][j]."""
    x, w = np.polynomial.legendre.leggauss(96)
    leg = _t(np.stack([w * np.polynomial.legendre.Legendre.basis(L)(x) for L in range(lmax + 1)], axis=1))
    x = _t(x)
    out = torch.empty((3, lmax + 1, len(pa), len(pb)), dtype=F64, device=DEV)
    step = max(1, (1 << 25) // (96 * len(pb)))
    for i in range(0, len(pa), step):
        p = pa[i:i + step, None, None]
        d = p * p + pb[None, :, None] ** 2 - 2.0 * p * pb[None, :, None] * x
        for k in range(3):
            out[k, :, i:i + step] = 2.0 * math.pi * torch.matmul(1.0 / (d + float(W.YUKAWA_PARAMS[k]) ** 2), leg).permute(2, 0, 1)
    return out


def _yukawa_terms(ch, lp, l, pa, pb, ints):
    """The 15 terms (V0 and 14 unit terms) of one l-block at the momenta pa x pb."""
    g, s, J = W.YUKAWA_PARAMS, ch.s, ch.J
    p, q = pa[:, None], pb[None, :]
    zero = torch.zeros((len(pa), len(pb)), dtype=F64, device=DEV)
    one = zero + 1.0
    u = [zero] * 14
    if lp == l:
        ls = 0.5 * (J * (J + 1.0) - l * (l + 1.0) - s * (s + 1.0))
        u[0] = ints[0, l]
        u[1] = (2.0 * s * (s + 1.0) - 3.0) * ints[0, l]
        u[2] = ints[1, l]
        u[3] = ls * p * q * (ints[1, l + 1] - (ints[1, l - 1] if l else 0.0)) / (2.0 * l + 1.0)
        if l == 0:
            u[5 + s], u[7 + s] = one, p * p + q * q
        if l == 1:
            at = {(1, 0): 9, (0, 1): 10, (1, 1): 11, (1, 2): 12}.get((s, J))
            if at:
                u[at] = p * q + zero
    if s == 1:
        if lp == l:
            t = 2.0 if l == J else (-2.0 * (J - 1.0) / (2.0 * J + 1.0) if l == J - 1 else -2.0 * (J + 2.0) / (2.0 * J + 1.0))
        else:
            t = 6.0 * math.sqrt(J * (J + 1.0)) / (2.0 * J + 1.0)
        u[4] = t * ints[2, (l + lp) // 2]
        if J == 1 and (lp, l) == (2, 0):
            u[13] = p * p + zero
        if J == 1 and (lp, l) == (0, 2):
            u[13] = q * q + zero
    reg = torch.exp(-(p * p + q * q) / float(g[3]) ** 2)
    u = [x * reg for x in u]
    v0 = sum(float(g[4 + k]) * u[k] for k in range(14))
    if s == 0 and l == 0 and ch.tz != 0:
        v0 = v0 + float(g[18]) * reg
    return torch.stack([v0] + u)


def _blocks(ch):
    return [ch.J - 1, ch.J + 1] if ch.coupled else [ch.l]


def _projected(c, N, chs):
    """Projected terms [T][n][n] of the channels that share the mesh of N bins."""
    kb, kq, om, norm, h0 = _mesh(N, c["wp_kind"])
    k, om = _t(kq), _t(om)
    bins = lambda v: (v * om[:, None] * om[None, :]).reshape(-1, N, W.MESH_Q, N, W.MESH_Q).sum((2, 4))  # noqa: E731
    got = []
    if c["pot"] == "yamaguchi":
        lam, beta = (float(x) for x in W.YAMAGUCHI_PARAMS)
        gk = 1.0 / (k * k + beta * beta)
        return [bins(lam * gk[:, None] * gk[None, :])[:1]]
    ints = _angle_integrals(k, k, max(max(_blocks(ch)) for ch in chs) + 1)
    for ch in chs:
        L = _blocks(ch)
        got.append(torch.cat([torch.cat([bins(_yukawa_terms(ch, a, b, k, k, ints)) for b in L], dim=2) for a in L], dim=1))
    return got


def _phases(T, q, K):
    """Phases in degrees [.., 3] of the continuum T [.., 2, 2] (complex) at momentum q."""
    g = 2.0 * math.pi * MU * q
    S = -1j * g[..., None, None] * T
    deg = 180.0 / math.pi
    out = torch.zeros(T.shape[:-2] + (3,), dtype=F64, device=DEV)
    d0 = 0.5 * torch.angle(1.0 + S[..., 0, 0])
    out[..., 0] = d0 * deg
    if K == 2:
        d1 = 0.5 * torch.angle(1.0 + S[..., 1, 1])
        x = (-1j * S[..., 0, 1] * torch.exp(-1j * (d0 + d1))).real
        out[..., 1] = d1 * deg
        out[..., 2] = 0.5 * torch.asin(x.clamp(-1.0, 1.0)) * deg
    return out


def _wrap(d):
    return d - 180.0 * torch.ceil((d - 90.0) / 180.0)


def _xlog(d):
    return torch.where(d == 0, torch.zeros_like(d), d * torch.log(d.abs()))


def _channel_T(V, cf, ch, mesh, wp_kind, e, point):
    """One channel, samples cf [S][T - 1]: T [S][m][2][2] at the needed bins (or energies) and the phases there."""
    kb, _, _, norm, h0 = mesh
    N, K = len(kb) - 1, ch.K
    n, S = K * N, (1 if cf is None else len(cf))
    H = V[:1].expand(S, n, n) if cf is None else V[0] + torch.einsum("st,tij->sij", cf, V[1:])
    Vs, h = H, _t(np.tile(h0, K))
    eps, C = _eigh(H + torch.diag(h))
    p = _momentum(e)
    kbt = _t(kb)
    mid = 0.5 * (kbt[1:] + kbt[:-1])
    pbin = (torch.searchsorted(kbt, p, right=True) - 1).clamp(0, N - 1)
    brk = (torch.searchsorted(mid, p, right=True) - 1).clamp(0, N - 2)
    if point:
        bins, q = pbin, p
    else:
        bins = torch.unique(torch.cat([pbin, brk, brk + 1]))
        q = mid[bins]
    T = torch.zeros((S, len(bins), 2, 2), dtype=torch.complex128, device=DEV)
    # samples with the same number of bound states share their packet layout
    nbs = (eps < 0).sum(1)
    step = max(1, (1 << 26) // (len(bins) * n))
    for nb in torch.unique(nbs).tolist():
        who = torch.nonzero(nbs == nb)[:, 0]
        for at in range(0, len(who), step):
            w = who[at:at + step]
            ep, Cw, Vw = eps[w], C[w], Vs[w]
            lo, hi = torch.empty_like(ep), torch.empty_like(ep)
            for start in range(K):  # the branches: every K-th positive state, dealt from the top
                idx = torch.arange(n - 1 - start, nb - 1, -K, device=DEV).flip(0)
                E = ep[:, idx]
                B = torch.cat([torch.zeros_like(E[:, :1]), 0.5 * (E[:, 1:] + E[:, :-1])], dim=1)
                top = E[:, -1:] + 0.5 * (B[:, -1:] - B[:, -2:-1])
                B = torch.cat([B, top], dim=1)
                lo[:, idx], hi[:, idx] = B[:, :-1], B[:, 1:]
            lo, hi, ep = lo[:, None], hi[:, None], ep[:, None]
            pos = torch.arange(n, device=DEV) >= nb
            if point:
                E = (p * p / (2.0 * MU))[None, :, None]
                re = torch.where(pos, torch.log(((E - lo) / (E - hi)).abs()) / (hi - lo), 1.0 / (E - ep))
                im = torch.where(pos & (E >= lo) & (E <= hi), -math.pi / (hi - lo), torch.zeros_like(re))
            else:
                a, b = (kbt[bins] ** 2 / (2.0 * MU))[None, :, None], (kbt[bins + 1] ** 2 / (2.0 * MU))[None, :, None]
                wd = (b - a) * (hi - lo)
                re = (_xlog(b - lo) - _xlog(a - lo) - _xlog(b - hi) + _xlog(a - hi)) / wd
                re = torch.where(pos, re, torch.log(((b - ep) / (a - ep)).abs()) / (b - a))
                ov = (torch.minimum(b, hi) - torch.maximum(a, lo)).clamp(min=0.0)
                im = torch.where(pos, -math.pi * ov / wd, torch.zeros_like(re))
            R = [torch.matmul(Vw[:, x * N + bins], Cw) for x in range(K)]
            for x in range(K):
                for y in range(K):
                    rr = R[x] * R[y]
                    T[w, :, x, y] = torch.complex((rr * re).sum(2) + Vw[:, x * N + bins, y * N + bins], (rr * im).sum(2))
    f2 = torch.ones_like(q) if wp_kind == W.WP_MOMENTUM else q / MU
    T = T * (f2 / (_t(norm)[bins] * q * q))[None, :, None, None]
    ph = _phases(T, q[None, :].expand(S, -1), K)
    if point:
        return T, ph
    at = lambda i: torch.searchsorted(bins, i)  # noqa: E731
    d0, d1 = ph[:, at(brk)], ph[:, at(brk + 1)].clone()
    d1[..., :2] += 180.0 * torch.round((d0[..., :2] - d1[..., :2]) / 180.0)
    wt = ((p - mid[brk]) / (mid[brk + 1] - mid[brk]))[None, :, None]
    d = d0 + wt * (d1 - d0)
    d[..., :2] = _wrap(d[..., :2])
    return T[:, at(pbin)], d


def _eigh(H):
    """Eigenpairs on the host's cores, one matrix per thread."""
    Hc = H.cpu()

    def one(M):
        torch.set_num_threads(1)
        return torch.linalg.eigh(M)

    with concurrent.futures.ThreadPoolExecutor(16) as ex:
        got = list(ex.map(one, Hc.unbind(0)))
    return torch.stack([g[0] for g in got]).to(H.device), torch.stack([g[1] for g in got]).to(H.device)


def _sigma(chs, delta, p):
    acc = torch.zeros((delta.shape[0], delta.shape[2]), dtype=F64, device=DEV)
    r = delta * (math.pi / 180.0)
    for k, ch in enumerate(chs):
        if ch.tz == 0:
            c2 = torch.cos(2.0 * r[:, k, :, 2])
            acc += (2.0 * ch.J + 1.0) * sum(1.0 - c2 * torch.cos(2.0 * r[:, k, :, b]) for b in range(ch.K))
    return math.pi / (2.0 * p * p) * 10.0 * acc


def _terms(c, sizes):
    got = [None] * len(sizes)
    chs = _channels(c)
    for N in sorted(set(sizes)):
        who = [k for k in range(len(chs)) if sizes[k] == N]
        for k, V in zip(who, _projected(c, N, [chs[k] for k in who])):
            got[k] = V
    return got


def _solve_exact(c, sizes, terms, cf, e):
    chs = _channels(c)
    cf, e = (None if cf is None else _t(cf)), _t(e)
    meshes = {N: _mesh(N, c["wp_kind"]) for N in set(sizes)}
    got = [_channel_T(terms[k], cf, chs[k], meshes[sizes[k]], c["wp_kind"], e, c["res"] == api.POINT) for k in range(len(chs))]
    delta = torch.stack([g[1] for g in got], dim=1)
    return torch.stack([g[0] for g in got], dim=1), delta, _sigma(chs, delta, _momentum(e))


def _mi_exact(c, seed):
    chs = _channels(c)
    cf, e = _draws(c, seed)
    cf, e = _t(cf), _t(e)
    x, w = np.polynomial.legendre.leggauss(c["n_quad"])
    th = math.pi * (1.0 + x) / 4.0
    kg, wg = _t(np.tan(th)), _t(math.pi / 4.0 * w / np.cos(th) ** 2)
    e_int = W.chebyshev_energies(c["n_int"])
    S, M = c["samples"], c["n_quad"] + 1
    Kon = torch.zeros((S, len(chs), c["n_int"], 2, 2), dtype=F64, device=DEV)
    ph = torch.zeros((S, len(chs), c["n_int"], 3), dtype=F64, device=DEV)
    lmax = max(max(_blocks(ch)) for ch in chs) + 1
    for i, p in enumerate(_momentum(_t(e_int))):
        q = torch.cat([kg, p[None]])
        den = p * p - kg * kg
        D = torch.cat([wg * kg * kg * 2.0 * MU / den, (-2.0 * MU * p * p * (wg / den).sum())[None]])
        ints = _angle_integrals(q, q, lmax)
        for k, ch in enumerate(chs):
            L = _blocks(ch)
            V = torch.cat([torch.cat([_yukawa_terms(ch, a, b, q, q, ints) for b in L], dim=2) for a in L], dim=1)
            V = V[0] + torch.einsum("st,tij->sij", cf, V[1:])
            cols = [M - 1 + b * M for b in range(ch.K)]
            A = torch.eye(ch.K * M, dtype=F64, device=DEV) - V * D.repeat(ch.K)
            X = torch.linalg.solve(A, V[:, :, cols])
            Kk = X[:, cols, :]
            Kon[:, k, i, :ch.K, :ch.K] = Kk
            T = torch.zeros((S, 2, 2), dtype=torch.complex128, device=DEV)
            one = torch.eye(ch.K, dtype=torch.complex128, device=DEV)
            T[:, :ch.K, :ch.K] = torch.linalg.solve(one + 1j * math.pi * MU * p * Kk, Kk.to(torch.complex128))
            ph[:, k, i] = _phases(T, p.expand(S), ch.K)
    et = _t(e_int)
    j = (torch.searchsorted(et, e, right=True) - 1).clamp(0, c["n_int"] - 2)
    wt = ((e - et[j]) / (et[j + 1] - et[j]))[None, None, :, None]
    d0, d1 = ph[:, :, j], ph[:, :, j + 1].clone()
    d1[..., :2] += 180.0 * torch.round((d0[..., :2] - d1[..., :2]) / 180.0)
    d = d0 + wt * (d1 - d0)
    for k, ch in enumerate(chs):
        d[:, k, :, :ch.K] = _wrap(d[:, k, :, :ch.K])
    return {"K": Kon, "delta": d, "sigma": _sigma(chs, d, _momentum(e))}


def _clebsch(j1, m1, j2, m2, J, Mz):
    if m1 + m2 != Mz or abs(m1) > j1 or abs(m2) > j2 or abs(Mz) > J or not abs(j1 - j2) <= J <= j1 + j2:
        return 0.0
    f = math.factorial
    pre = math.sqrt((2 * J + 1) * f(J + j1 - j2) * f(J - j1 + j2) * f(j1 + j2 - J) / f(j1 + j2 + J + 1)
                    * f(J + Mz) * f(J - Mz) * f(j1 - m1) * f(j1 + m1) * f(j2 - m2) * f(j2 + m2))
    tot = 0.0
    for k in range(j1 + j2 - J + 1):
        d = [k, j1 + j2 - J - k, j1 - m1 - k, j2 + m2 - k, J - j2 + m1 + k, J - j1 - m2 + k]
        if min(d) >= 0:
            tot += (-1) ** k / math.prod(f(x) for x in d)
    return pre * tot


def _ylm(l, m, x):
    """Y_l^m(theta, 0) at x = cos theta."""
    am = abs(m)
    if am > l:
        return torch.zeros_like(x)
    s = torch.sqrt(1.0 - x * x)
    pmm = torch.ones_like(x)
    for i in range(1, am + 1):
        pmm = pmm * (2 * i - 1) * s
    p0, p1 = torch.zeros_like(x), pmm
    for k in range(am + 1, l + 1):
        p0, p1 = p1, ((2 * k - 1) * x * p1 - (k + am - 1) * p0) / (k - am)
    y = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - am) / math.factorial(l + am)) * p1
    return -y if m > 0 and am % 2 else y


def _spin_exact(c, seed):
    chs = _channels(c)
    d, e, th = (_t(x) for x in _draws(c, seed))
    p = _momentum(e)[None, :, None]
    r = d * (math.pi / 180.0)
    x = torch.cos(th)
    S, nE, nT = c["samples"], c["energies"], c["angles"]
    M = {(s, a, b): torch.zeros((S, nE, nT), dtype=torch.complex128, device=DEV)
         for s in (0, 1) for a in range(-s, s + 1) for b in range(-s, s + 1)}
    for k, ch in enumerate(chs):
        dm, dp, ep = r[:, k, :, 0], r[:, k, :, 1], r[:, k, :, 2]
        L = _blocks(ch)
        if ch.K == 1:
            Sm = {(0, 0): torch.exp(2j * dm)}
        else:
            off = 1j * torch.sin(2 * ep) * torch.exp(1j * (dm + dp))
            Sm = {(0, 0): torch.cos(2 * ep) * torch.exp(2j * dm), (1, 1): torch.cos(2 * ep) * torch.exp(2j * dp),
                  (0, 1): off, (1, 0): off}
        for (a, b), v in Sm.items():
            amp = v - 1.0 if a == b else v
            for mp in range(-ch.s, ch.s + 1):
                for m in range(-ch.s, ch.s + 1):
                    w = math.sqrt(4 * math.pi) * math.sqrt(2 * L[b] + 1) * _clebsch(L[a], m - mp, ch.s, mp, ch.J, m) \
                        * _clebsch(L[b], 0, ch.s, m, ch.J, m)
                    if w:
                        M[ch.s, mp, m] += w * amp[:, :, None] * _ylm(L[a], m - mp, x)[None, None, :]
    M = {k: v / (2j * p) for k, v in M.items()}
    # to the product basis uu, ud, du, dd
    h = math.sqrt(0.5)
    vec = {(1, 1): [1, 0, 0, 0], (1, 0): [0, h, h, 0], (1, -1): [0, 0, 0, 1], (0, 0): [0, h, -h, 0]}
    full = torch.zeros((S, nE, nT, 4, 4), dtype=torch.complex128, device=DEV)
    for (s, a, b), v in M.items():
        full += v[..., None, None] * torch.tensor(np.outer(vec[s, a], vec[s, b]), dtype=torch.complex128, device=DEV)
    pauli = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=torch.complex128, device=DEV)
    ch2, sh2, z = torch.cos(0.5 * th), torch.sin(0.5 * th), torch.zeros_like(th)
    along = lambda v: torch.einsum("vt,vij->tij", torch.stack(v).to(torch.complex128), pauli)  # noqa: E731
    Pl, Pm, Pn = along([sh2, z, ch2]), along([-ch2, z, sh2]), along([z, z + 1, z])
    one = torch.eye(2, dtype=torch.complex128, device=DEV).expand(nT, 2, 2)
    kron = lambda A, B: torch.einsum("tij,tkl->tikjl", A, B).reshape(nT, 4, 4)  # noqa: E731
    tr = lambda O: torch.einsum("setij,tji->set", full, O)  # noqa: E731
    apb, amb = 0.5 * tr(kron(one, one)), 0.5 * tr(kron(Pn, Pn))
    cpd, cmd = 0.5 * tr(kron(Pm, Pm)), 0.5 * tr(kron(Pl, Pl))
    ee = 0.25 * (tr(kron(Pn, one)) + tr(kron(one, Pn)))
    amps = torch.stack([0.5 * (apb + amb), 0.5 * (apb - amb), 0.5 * (cpd + cmd), 0.5 * (cpd - cmd), ee], dim=-1)
    return {"abcde": torch.view_as_real(amps), "dsig": 2.5 * (full.abs() ** 2).sum((-1, -2))}


def exact(case, seed):
    c = case
    if c["kind"] == "spin":
        return _spin_exact(c, seed)
    if c["kind"] == "mi":
        return _mi_exact(c, seed)
    sizes = _sizes(c)
    if c["kind"] == "serve":
        choices = [int(x) for x in c["n_wp"].split(",")]
        reqs = _draws(c, seed)
        terms = {N: _terms(c, [N] * len(sizes)) for N in choices}
        got = [_solve_exact(c, [n] * len(sizes), terms[n], cf[None], e) for cf, e, n in reqs]
        cat = lambda k: torch.cat([g[k].reshape(-1) for g in got]).cpu().numpy()  # noqa: E731
        return {"T": cat(0), "delta": cat(1), "sigma": cat(2), "status": None}
    if c["samples"] * sum((ch.K * n) ** 3 for ch, n in zip(_channels(c), sizes)) > 3e10:
        return None  # minutes of host eigendecompositions
    cf, e = _draws(c, seed)
    T, d, s = _solve_exact(c, sizes, _terms(c, sizes), cf, e)
    got = {"T": torch.view_as_real(T), "delta": d, "sigma": s}
    return {k: v.cpu().numpy() for k, v in got.items()} if c["kind"] == "host" else got
