"""Sizes and batch shapes at which a solve changes its route.

* FP64 T: V C rows from the tensor cores from n = 80 on, explicit below, shares of
  the bins over several CTAs: around that size and the products' tiles (64, 128),
  with energies that fill one share or leave the last one ragged, both kinds of
  resolvent, against the oracle at the FP64 tolerances.
* FP32 Jacobi: one team of warps below n = 160, two from there to n = 304, global
  memory above: mixed solves around both limits against the oracle at the mixed ones.
* Small batches run their size buckets on several streams, and a large matrix on
  a cluster of as many CTAs as are free: the same samples one after another
  (profiling), alone and in a larger batch give the same bits."""
import dataclasses

import numpy as np
import pytest

from paper_2106_00454_gb300 import inputs as W

from parity_util import compare, compare_mixed, gpu_run, oracle_run

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


def _wl(channels, n_wp, S, n_e, lo=2.0, hi=300.0, wp_kind=W.WP_MOMENTUM):
    return W.Workload("paths", channels, [n_wp] * len(channels), W.GEN_YUKAWA, W.YUKAWA_PARAMS.copy(), W.N_TERMS_YUKAWA,
                      W.coefficient_samples(S, 11), np.linspace(lo, hi, n_e), wp_kind=wp_kind)


UNC, CPL = W.Channel(0, 0, 0, 0, 0), W.Channel(1, 1, 0, 2, 1)


@pytest.mark.parametrize("ch,n_wp", [(UNC, 79), (UNC, 80), (CPL, 39), (CPL, 40), (UNC, 64), (UNC, 65), (CPL, 64), (CPL, 65)],
                         ids=lambda x: x if isinstance(x, int) else x.name)
@pytest.mark.parametrize("n_e,res", [(1, 0), (50, 0), (2, 2), (33, 2)])
def test_fp64_t_routes(ctx, orc, ch, n_wp, n_e, res):
    from paper_2106_00454_gb300 import api
    wl = _wl([ch], n_wp, 2, n_e, wp_kind=W.WP_ENERGY if res else W.WP_MOMENTUM)
    md = api.Model(ctx, wl)
    compare(wl, gpu_run(ctx, md, wl, res=res), oracle_run(orc, wl, mode=res))


@pytest.mark.parametrize("ch,n_wp", [(UNC, 159), (UNC, 160), (UNC, 161), (CPL, 80), (CPL, 152), (CPL, 153)],
                         ids=lambda x: x if isinstance(x, int) else x.name)
def test_mixed_kernel_limits(ctx, orc, ch, n_wp):
    from paper_2106_00454_gb300 import api
    wl = _wl([ch], n_wp, 2, 9)
    md = api.Model(ctx, wl)
    compare_mixed(wl, gpu_run(ctx, md, wl, prec=1), oracle_run(orc, wl))


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_buckets_on_streams_same_bits(ctx, prec):
    from paper_2106_00454_gb300 import api
    wl = W.workload_batched(n_samples=5, n_e=21, nwp_choices=(21, 30, 41, 52))
    md = api.Model(ctx, wl)
    gpu_run(ctx, md, wl, prec=prec)  # the autotuner's calls
    a = [gpu_run(ctx, md, wl, prec=prec) for _ in range(2)]
    ctx.profile(True)
    try:
        b = gpu_run(ctx, md, wl, prec=prec)
    finally:
        ctx.profile(False)
    for r in a:
        for x, y in zip(r, b):
            assert np.array_equal(x, y)


def test_large_matrices_same_bits_alone_and_in_a_batch(ctx):
    from paper_2106_00454_gb300 import api
    wl = _wl([CPL], 160, 80, 7)
    md = api.Model(ctx, wl)
    whole = gpu_run(ctx, md, wl, prec=1)
    for s, k in ((3, 1), (0, 20), (10, 40)):  # clusters of 8, 4 or less, 2 or less
        part = gpu_run(ctx, md, dataclasses.replace(wl, coeffs=wl.coeffs[s:s + k]), prec=1)
        for x, y in zip(part, whole):
            assert np.array_equal(x, y[s:s + k])


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_one_solve_per_launch_same_bits(ctx, prec):
    """Plain execution of several channels of one size (each its own mean-potential basis)."""
    from paper_2106_00454_gb300 import api
    wl = _wl([UNC, W.Channel(1, 1, 1, 1, 0), CPL, W.Channel(1, 2, 1, 3, 1)], 32, 2, 9)
    md = api.Model(ctx, wl)
    a = gpu_run(ctx, md, wl, prec=prec)
    ctx.set_exec(api.EXEC_PLAIN)
    try:
        b = gpu_run(ctx, md, wl, prec=prec)
    finally:
        ctx.set_exec(api.EXEC_BATCHED)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_sample_ranges_same_bits(ctx):
    """One size bucket above a stream's share of the scratch goes in sample ranges."""
    from paper_2106_00454_gb300 import api
    wl = _wl([CPL], 100, 2500, 3)
    md = api.Model(ctx, wl)
    gpu_run(ctx, md, dataclasses.replace(wl, coeffs=wl.coeffs[:2]), prec=1)
    whole = gpu_run(ctx, md, wl, prec=1)
    for s in (0, 1240, 1250, 2490):
        part = gpu_run(ctx, md, dataclasses.replace(wl, coeffs=wl.coeffs[s:s + 10]), prec=1)
        for x, y in zip(part, whole):
            assert np.array_equal(x, y[s:s + 10])


def test_no_room_for_the_streams_same_bits(ctx):
    """A budget that holds one bucket's scratch at a time, not a share for each stream."""
    import torch
    from paper_2106_00454_gb300 import api
    wl = W.workload_batched(n_samples=40, n_e=9, nwp_choices=(30, 31, 32, 33))
    S, nch = 40, len(wl.channels)

    def phases(c, md, n):
        cf = torch.tensor(wl.coeffs, dtype=torch.float64, device="cuda:0")
        e = torch.tensor(wl.e_lab, dtype=torch.float64, device="cuda:0")
        d = torch.zeros((S, nch, 9, 3), dtype=torch.float64, device="cuda:0")
        for _ in range(n):
            c.solve(md.vset, cf, S, e, None, d, None, prec=1)
            c.sync()
        return d.cpu().numpy()

    probe = api.Context(0)
    md = api.Model(probe, wl)
    probe.profile(True)  # one bucket after another
    phases(probe, md, 2)
    room = probe.bytes_in_use() + (1 << 20)
    probe.close()
    tight = api.Context(0, hbm_budget_bytes=room)
    a = phases(tight, api.Model(tight, wl), 4)
    assert tight.bytes_in_use() <= room
    tight.close()
    assert np.array_equal(a, phases(ctx, api.Model(ctx, wl), 3))


@pytest.mark.parametrize("nq,S", [(24, 60), (33, 41)])
def test_inversion_side_by_side_same_bits(ctx, nq, S):
    """Both block sizes of an inversion on two streams (once their kernels are tuned),
    against one after the other (profiling)."""
    from test_gpu_mi import _gpu
    chs = [c.astuple() for c in W.np_channels(2)]
    coeffs, e_lab, e_int = W.coefficient_samples(S, 6), W.lab_energies(9), W.chebyshev_energies(14)
    args = (chs, W.GEN_YUKAWA, W.YUKAWA_PARAMS, W.N_TERMS_YUKAWA, coeffs, e_int, e_lab, nq)
    assert S * len(chs) * 14 >= 12 * 152
    runs = [_gpu(ctx, *args) for _ in range(3)]
    ctx.profile(True)
    try:
        runs.append(_gpu(ctx, *args))
    finally:
        ctx.profile(False)
    for r in runs[1:]:
        for x, y in zip(r, runs[0]):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("ch,n_wp", [(UNC, 15), (UNC, 33), (CPL, 64)], ids=lambda x: x if isinstance(x, int) else x.name)
def test_fp64_update_shared_by_ctas_same_bits(ctx, ch, n_wp):
    """The refinement's update: one CTA a matrix in a large batch, up to eight in a small one."""
    from paper_2106_00454_gb300 import api
    wl = _wl([ch], n_wp, 1300, 5)
    md = api.Model(ctx, wl)
    whole = gpu_run(ctx, md, wl)
    for s, k in ((7, 1), (100, 60), (300, 130)):
        part = gpu_run(ctx, md, dataclasses.replace(wl, coeffs=wl.coeffs[s:s + k]))
        for x, y in zip(part, whole):
            assert np.array_equal(x, y[s:s + k])
