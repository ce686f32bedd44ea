"""Levels whose large entities are split over CTAs, at the edges of the layout.

HIFCN_SPLIT_DOFS=1 sends every level with an entity of more than 32 DOFs there:
inputs gathered by four CTAs per entity (256 DOFs a pass) with the level's small
entities in the same launch, rows of H by blocks of 32, columns by blocks of 64
with 16 row groups.  eps = 0 keeps the entities whole: 33 to 121 DOFs in 3D, 31
to 129 in 2D, with small ones beside them and without.

Bars: the apply of the same imported factor within 1e-12 (FP64), 1e-5 (FP32) and
3e-2 (BF16 top levels) of the oracle, the bars of these applies everywhere.
"""

import numpy as np
import pytest

import workloads as W
from parity import rel_err
from oracle import export, grid, hif

pytestmark = pytest.mark.gpu

CASES = [(2, 64, 16), (2, 68, 17), (2, 130, 65), (2, 132, 33), (3, 12, 6), (3, 16, 4), (3, 24, 6)]


@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_n{n}_m{m}" for d, n, m in CASES])
def test_split_entities_apply(case, monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    monkeypatch.setenv("HIFCN_SPLIT_DOFS", "1")
    monkeypatch.setenv("HIFCN_NO_LEVEL_FUSE", "1")
    dim, n, m = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=0.0, contrast=1e2, dt=0.1, seed=9)
    F = hif.factor(grid.assemble_A(w.a_nodes, w.dt), n, dim, m, 0.0)
    x = np.random.default_rng(10).standard_normal(F.N)
    ref = hif.apply_inverse(F, x)
    xt = torch.from_numpy(x).cuda()
    blob = export.export_blob(F, w.dt)
    for prec, bars in ((H.HIF_FP32, {None: 1e-12, H.HIF_FP32: 1e-5}), (H.HIF_FP32_BF16TOP, {H.HIF_FP32_BF16TOP: 3e-2})):
        h = H.hif_import_factor(dim, n, m, blob, w.dt, torch.from_numpy(w.a_nodes).cuda(),
                                H.default_options(eps=0.0, precision=prec))
        for p, bar in bars.items():
            y = H.hif_apply(h, xt) if p is None else H.hif_apply(h, xt, precision=p)
            assert rel_err(y.cpu().numpy(), ref) <= bar
        h.close()
