"""Tuning the cell cuts does not take levels out of the fused launches.

The tuner times the levels in launches of their own; a cut that is faster there may
leave a level's cells whole, which moves it to the S-form kernels and ends the range
of the fused ones, whose apply is the faster.

Bars: the fused launches of an FP32 apply before tuning are all there after it, and
the apply is that of before within 1e-5 (FP32 rounding in another order).
"""

import pytest

import workloads as W

pytestmark = pytest.mark.gpu

CASES = [(2, 128, 4, 1e-3), (2, 256, 8, 1e-6), (2, 352, 11, 1e-6), (2, 704, 11, 1e-3)]


@pytest.mark.parametrize("case", CASES, ids=[f"n{n}_m{m}" for _, n, m, _ in CASES])
def test_fused_range_survives_tuning(case):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m, eps = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=eps, contrast=1e2, dt=0.1, seed=41)
    h = H.hif_setup(dim, n, m, torch.from_numpy(w.a_nodes).cuda(), w.dt,
                    H.default_options(eps=eps, precision=H.HIF_FP32))
    x = torch.randn(w.N, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))

    def apply():
        H.hif_stats_enable(h, True)
        y = H.hif_apply(h, x, precision=H.HIF_FP32)
        names = {r["name"] for r in H.hif_stats_read(h) if r["name"].startswith("level_")}
        H.hif_stats_enable(h, False)
        return y, names

    y0, before = apply()
    assert "level_fwd_l3" in before
    H.hif_autotune(h)
    y1, after = apply()
    assert before <= after, before - after
    assert float((y1 - y0).norm()) <= 1e-5 * float(y0.norm())
    h.close()
