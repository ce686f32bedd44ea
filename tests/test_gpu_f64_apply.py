"""FP64 apply at the edges of its cell kernels' layouts.

The forward step takes a row of a cell per eight lanes (pairs of columns, four
rows a warp), the backward step blocks of 32 columns, 256 at a time, with the
rows spread over the warps.  The leaf sizes put the interiors (leaf - 1)^dim
just below, at and above those edges: 1, 16, 25, 216, 256, 289 and 343 DOFs,
with boundaries of a few to several hundred DOFs; cells whole and cut into
items.

Bar: 1e-12 of the oracle's apply on the same (imported) factor, the bar of the
FP64 apply everywhere: sums of at most a few hundred products in another order,
a few stages deep.
"""

import numpy as np
import pytest

import workloads as W
from parity import rel_err
from oracle import export, grid, hif

pytestmark = pytest.mark.gpu

CASES = [(2, 8, 2), (2, 20, 5), (2, 24, 6), (2, 34, 17), (2, 36, 18), (3, 14, 7), (3, 16, 8)]


@pytest.mark.parametrize("target", ["1", "0"], ids=["whole", "cut"])
@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_n{n}_m{m}" for d, n, m in CASES])
def test_f64_apply_at_layout_edges(case, target, monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    if target != "0":
        monkeypatch.setenv("HIFCN_ITEM_TARGET", target)
    dim, n, m = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=1e-6, contrast=1e2, dt=0.1, seed=5)
    F = hif.factor(grid.assemble_A(w.a_nodes, w.dt), n, dim, m, 1e-6)
    h = H.hif_import_factor(dim, n, m, export.export_blob(F, w.dt), w.dt,
                            torch.from_numpy(w.a_nodes).cuda(), H.default_options(eps=1e-6))
    x = np.random.default_rng(2).standard_normal(F.N)
    y = H.hif_apply(h, torch.from_numpy(x).cuda()).cpu().numpy()
    assert rel_err(y, hif.apply_inverse(F, x)) <= 1e-12
    h.close()
