"""The autotuner's choice for a matrix size comes from a batch that a caller sent."""
import numpy as np
import pytest

from paper_2106_00454_gb300 import inputs as W

pytestmark = pytest.mark.gpu


def test_fp64_choice_is_timed_on_the_first_batch():
    """A set with sample terms is solved at its mean first (one matrix, the start
    basis).  That solve must not fix the CTA size: the table's time per solve is
    that of the batch, as without a start basis, where a matrix alone on the chip
    takes about a hundred times as long as its share of a full wave (152 SMs)."""
    import torch
    from paper_2106_00454_gb300 import api, build
    build.build()
    S, N = 1300, 40
    wl = W.Workload("tune", [W.Channel(0, 0, 0, 0, 0)], [N], W.GEN_YUKAWA, W.YUKAWA_PARAMS.copy(), W.N_TERMS_YUKAWA,
                    W.coefficient_samples(S, 3), np.linspace(2.0, 300.0, 5))
    best = []
    for rotate in (False, True):
        ctx = api.Context(0)
        ctx.set_rotate(rotate)
        md = api.Model(ctx, wl)
        cf = torch.tensor(wl.coeffs, dtype=torch.float64, device="cuda:0")
        e = torch.tensor(wl.e_lab, dtype=torch.float64, device="cuda:0")
        d = torch.zeros((S, 1, 5, 3), dtype=torch.float64, device="cuda:0")
        ctx.solve(md.vset, cf, S, e, None, d, None)
        ctx.sync()
        (entry,) = [x for x in ctx.tuning() if x["n"] == N and x["precision"] == "fp64"]
        best.append(entry["ms_per_solve"][entry["threads"]])
        ctx.close()
    assert best[1] <= 8.0 * best[0], best
