"""Fused upper levels of the FP32 apply against the oracle.

The fused launches form an entity step and the next level's cell step in one CTA
(positions concatenated per cell, first rows preloaded, two vectors in turn).
Leaf sizes and depths put entities at 1 to 33 DOFs, cells beside 128 interior
DOFs, one to six levels, CTAs of 256 and 512 threads, and 3D levels with small
faces; eps = 0.5 leaves entities without surviving DOFs.

Bars: the FP32 apply within 1e-5 of the oracle on the same imported factor, and
equal to the per-level launches (HIFCN_NO_LEVEL_FUSE=1) within 1e-5; the same call
gives the same bits; the statistics name the fused launches.
"""

import numpy as np
import pytest

import workloads as W
from parity import rel_err
from oracle import export, grid, hif

pytestmark = pytest.mark.gpu

CASES = [(2, 8, 4, 1e-6), (2, 8, 2, 1e-6), (2, 16, 2, 0.0), (2, 32, 16, 1e-6), (2, 36, 9, 0.5), (2, 64, 8, 1e-6),
         (2, 128, 4, 1e-3), (2, 132, 33, 1e-6), (2, 128, 32, 0.0), (2, 128, 16, 1e-8), (2, 320, 10, 1e-3),
         (3, 8, 4, 1e-4), (3, 16, 4, 0.5), (3, 12, 3, 1e-2)]


@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_n{n}_m{m}_eps{e:g}" for d, n, m, e in CASES])
def test_fused_levels_apply(case, monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m, eps = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=eps, contrast=1e2, dt=0.1, seed=12)
    F = hif.factor(grid.assemble_A(w.a_nodes, w.dt), n, dim, m, eps)
    blob = export.export_blob(F, w.dt)
    a = torch.from_numpy(w.a_nodes).cuda()
    opt = H.default_options(eps=eps, precision=H.HIF_FP32)
    x = np.random.default_rng(3).standard_normal(F.N)
    xt = torch.from_numpy(x).cuda()
    h = H.hif_import_factor(dim, n, m, blob, w.dt, a, opt)
    H.hif_stats_enable(h, True)
    H.hif_apply(h, xt, precision=H.HIF_FP32)
    assert any(r["name"].startswith("level_top") for r in H.hif_stats_read(h))
    H.hif_stats_enable(h, False)
    y = H.hif_apply(h, xt, precision=H.HIF_FP32)
    assert torch.equal(y, H.hif_apply(h, xt, precision=H.HIF_FP32))
    assert rel_err(y.cpu().numpy(), hif.apply_inverse(F, x)) <= 1e-5
    monkeypatch.setenv("HIFCN_NO_LEVEL_FUSE", "1")
    h1 = H.hif_import_factor(dim, n, m, blob, w.dt, a, opt)
    assert rel_err(y.cpu().numpy(), H.hif_apply(h1, xt, precision=H.HIF_FP32).cpu().numpy()) <= 1e-5
    h.close()
    h1.close()
