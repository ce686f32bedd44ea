"""Multi-column apply: the FP32 levels' kernel at the edges of its tiles.

The kernel takes 128-row tiles, K in chunks of 32 (a backward cell's V rows
start on a multiple of 64) and columns by 8, 16 or 32.  Leaf interiors of 1,
25, 225, 256, 289 and 343 DOFs and k at and beside the column tiles; with
HIFCN_ITEM_TARGET=1 the 2D leaf level is one that the single-column apply runs
in the S-form, whose backward step the kernel replaces by its compensated form.

Bars, as for the BF16 levels' kernel: every column within 3e-2 of the oracle
(BF16 root) and within 1e-3 of the single-column apply of the same handle.
"""

import numpy as np
import pytest

import workloads as W
from parity import rel_err
from oracle import export, grid, hif

pytestmark = pytest.mark.gpu

CASES = [(2, 8, 2, 0), (2, 24, 6, 0), (2, 64, 16, 1), (2, 68, 17, 1), (2, 36, 18, 0), (3, 16, 8, 0)]
_cache = {}


@pytest.mark.parametrize("k", [1, 8, 9, 17, 64])
@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_n{n}_m{m}{'_whole' * t}" for d, n, m, t in CASES])
def test_fp32_levels_at_tile_edges(case, k, monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m, whole = case
    if whole:
        monkeypatch.setenv("HIFCN_ITEM_TARGET", "1")
    if case not in _cache:
        w = W.small_variable_2d(n=n, m=m, dim=dim, eps=1e-6, contrast=1e2, dt=0.1, seed=9)
        F = hif.factor(grid.assemble_A(w.a_nodes, w.dt), n, dim, m, 1e-6)
        _cache[case] = (w, F, export.export_blob(F, w.dt))
    w, F, blob = _cache[case]
    levels = len(F.level_factors)
    h = H.hif_import_factor(dim, n, m, blob, w.dt, torch.from_numpy(w.a_nodes).cuda(),
                            H.default_options(eps=1e-6, precision=H.HIF_FP32_BF16TOP,
                                              bf16_top_levels=max(1, levels - 1)))
    X = np.random.default_rng(k).standard_normal((k, w.N))
    Y = H.hif_apply_multi(h, torch.from_numpy(X).cuda()).cpu().numpy()
    for c in sorted({0, k // 2, k - 1}):
        single = H.hif_apply(h, torch.from_numpy(X[c].copy()).cuda(),
                             precision=H.HIF_FP32_BF16TOP).cpu().numpy()
        assert rel_err(Y[c], hif.apply_inverse(F, X[c])) <= 3e-2
        assert rel_err(Y[c], single) <= 1e-3
    h.close()
