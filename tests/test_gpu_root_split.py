"""The split root and the FP32 backward cells at the edges of their layouts.

Roots are applied by rows and by blocks of 128 columns x 128 rows
(HIFCN_ROOT_SPLIT_DOFS=1 sends every root there): roots of 3 to 45, 125, 129 and 631
DOFs around those edges.  The FP32 backward step takes blocks of at most 32
column quads: interiors of 1, 25, 121, 256, 289 and 343 DOFs, whole and cut.

Bars: the apply of the same imported factor within 1e-12 (FP64) and 1e-5 (FP32)
of the oracle, the bars of these applies everywhere.
"""

import numpy as np
import pytest

import workloads as W
from parity import rel_err
from oracle import export, grid, hif

pytestmark = pytest.mark.gpu

# (dim, n, leaf), eps = 0: the root is the top separator, 2 (n - 1) - 1 DOFs in 2D
CASES = [(2, 4, 2), (2, 8, 4), (2, 24, 12), (2, 64, 32), (2, 66, 33), (2, 128, 8),
         (3, 14, 7), (3, 16, 8), (2, 34, 17), (2, 36, 18)]


@pytest.mark.parametrize("target", ["1", "0"], ids=["whole", "cut"])
@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_n{n}_m{m}" for d, n, m in CASES])
def test_split_root_apply(case, target, monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    monkeypatch.setenv("HIFCN_ROOT_SPLIT_DOFS", "1")
    if target != "0":
        monkeypatch.setenv("HIFCN_ITEM_TARGET", target)
        monkeypatch.setenv("HIFCN_NO_TMA", "1")
    dim, n, m = case
    eps = 0.0 if n < 100 or m > 8 else 1e-3
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=eps, contrast=1e2, dt=0.1, seed=6)
    F = hif.factor(grid.assemble_A(w.a_nodes, w.dt), n, dim, m, eps)
    h = H.hif_import_factor(dim, n, m, export.export_blob(F, w.dt), w.dt, torch.from_numpy(w.a_nodes).cuda(),
                            H.default_options(eps=eps, precision=H.HIF_FP32))
    x = np.random.default_rng(8).standard_normal(F.N)
    ref = hif.apply_inverse(F, x)
    xt = torch.from_numpy(x).cuda()
    assert rel_err(H.hif_apply(h, xt).cpu().numpy(), ref) <= 1e-12
    assert rel_err(H.hif_apply(h, xt, precision=H.HIF_FP32).cpu().numpy(), ref) <= 1e-5
    # the ticket counters are back at zero: the same call gives the same bits
    assert torch.equal(H.hif_apply(h, xt), H.hif_apply(h, xt))
    h.close()
