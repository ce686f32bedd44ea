"""The block-Jacobi scaling of the fronts at the edges of its 32 x 32 tiles.

At eps = 0 nothing is skeletonized away, so the factor is exact whatever the
scaling: leaf sizes giving boundaries of 12 to 366 DOFs (tiles partly filled, a
full one, many), 2D and 3D, in one chunk of cells and in one-cell chunks.

Bars: the apply is the inverse to 1e-9 of the right-hand side (the bar of the
exact factor in these tests), and the chunked setup gives the same bits.
"""

import numpy as np
import pytest

import workloads as W
from oracle import grid

pytestmark = pytest.mark.gpu

CASES = [(2, 8, 4), (2, 16, 8), (2, 36, 9), (2, 66, 33), (3, 8, 4), (3, 16, 8), (3, 18, 9)]


@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_n{n}_m{m}" for d, n, m in CASES])
def test_scaled_fronts(case, monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=0.0, contrast=1e2, dt=0.1, seed=12)
    A = grid.assemble_A(w.a_nodes, w.dt)
    x = np.random.default_rng(13).standard_normal(A.shape[0])
    b = torch.from_numpy(A @ x).cuda()
    ys = []
    for chunk in (None, "1"):
        if chunk:
            monkeypatch.setenv("HIFCN_SETUP_SCRATCH_BYTES", chunk)
        h = H.hif_setup(dim, n, m, torch.from_numpy(w.a_nodes).cuda(), w.dt, H.default_options(eps=0.0))
        ys.append(H.hif_apply(h, b))
        h.close()
    assert np.linalg.norm(ys[0].cpu().numpy() - x) <= 1e-9 * np.linalg.norm(x)
    assert torch.equal(ys[0], ys[1])
