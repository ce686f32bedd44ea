"""The FP64 apply of small roots from shared memory.

Roots of at most 212 DOFs are copied to shared memory before the apply reaches
them; larger ones are read in place.  Roots of 5 to 205 DOFs on the first path,
around its 32-column groups, and of 213 and 221 on the second.

Bar: 1e-12 of the oracle's apply on the same (imported) factor, the bar of the
FP64 apply everywhere.
"""

import numpy as np
import pytest

import workloads as W
from parity import rel_err
from oracle import export, grid, hif

pytestmark = pytest.mark.gpu

# (n, leaf), eps = 0: the root is the top separator, 2 (n - 1) - 1 DOFs
CASES = [(4, 2), (16, 8), (18, 9), (34, 17), (64, 16), (66, 33), (104, 13), (108, 27), (112, 14)]


@pytest.mark.parametrize("case", CASES, ids=[f"n{n}_m{m}" for n, m in CASES])
def test_f64_root(case):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    n, m = case
    w = W.small_variable_2d(n=n, m=m, dim=2, eps=0.0, contrast=1e2, dt=0.1, seed=4)
    F = hif.factor(grid.assemble_A(w.a_nodes, w.dt), n, 2, m, 0.0)
    h = H.hif_import_factor(2, n, m, export.export_blob(F, w.dt), w.dt, torch.from_numpy(w.a_nodes).cuda(),
                            H.default_options(eps=0.0))
    x = np.random.default_rng(3).standard_normal(F.N)
    xt = torch.from_numpy(x).cuda()
    y = H.hif_apply(h, xt)
    assert rel_err(y.cpu().numpy(), hif.apply_inverse(F, x)) <= 1e-12
    assert torch.equal(H.hif_apply(h, xt), y)
    h.close()
