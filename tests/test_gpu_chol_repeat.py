"""The factorization of the diagonal blocks gives the same bits on every run.

Panels of 1 to 32 columns (interiors of 5 to 125 DOFs above the leaf level, roots of
29 to 331), many cells and one.  Bars: exported factors equal byte for byte over
repeated setups, and A applied to F^{-1} b gives b back within 1e-9 (eps = 0).
"""

import numpy as np
import pytest

import workloads as W
from oracle import grid

pytestmark = pytest.mark.gpu

CASES = [(2, 16, 2), (2, 32, 8), (2, 64, 4), (2, 128, 16), (2, 68, 17), (3, 12, 3)]


@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_n{n}_m{m}" for d, n, m in CASES])
def test_same_bits(case):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=0.0, contrast=1e2, dt=0.2, seed=7)
    a = torch.from_numpy(w.a_nodes).cuda()
    x = np.random.default_rng(8).standard_normal(w.N)
    b = torch.from_numpy(grid.assemble_A(w.a_nodes, w.dt) @ x).cuda()
    blobs = []
    for _ in range(4):
        h = H.hif_setup(dim, n, m, a, w.dt, H.default_options(eps=0.0))
        blobs.append(H.hif_export_factor(h))
        y = H.hif_apply(h, b).cpu().numpy()
        assert np.linalg.norm(y - x) <= 1e-9 * np.linalg.norm(x)
        h.close()
    assert all(v == blobs[0] for v in blobs)
