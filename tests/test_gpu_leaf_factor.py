"""Leaf elimination from the stencil at the edges of its layout.

The kernel takes a cell's band of half width (leaf - 1)^(dim - 1) in buffers of
8, 16, 32 or 64 values and 32 columns a warp; wider bands (2D leaf 34: its band
does not fit shared memory, 3D leaf 10) take the dense fronts.  With eps = 0 the
factor is exact, so F^{-1} A x = x up to rounding: within 1e-9 (A >= I and
||A|| < 1e6 here, so the condition times rounding is 1e-10); the leaf operators G
and V of the factor blob against dense algebra in FP64 within 1e-11 of their norms
(condition of a leaf block, below 1e4, times rounding, with a margin of ten).
"""

import numpy as np
import pytest

import workloads as W
from blobutil import read_blob
from oracle import grid

pytestmark = pytest.mark.gpu

# dim, n, leaf
CASES = [(2, 8, 2), (2, 18, 9), (2, 20, 10), (2, 34, 17), (2, 36, 18), (2, 54, 27), (2, 68, 34),
         (3, 8, 4), (3, 10, 5), (3, 12, 6), (3, 18, 9), (3, 20, 10)]


@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_m{m}" for d, n, m in CASES])
def test_leaf_factor(case, monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=0.0, contrast=1e3, dt=0.5, seed=3)
    A = grid.assemble_A(w.a_nodes, w.dt)
    a = torch.from_numpy(w.a_nodes).cuda()
    h = H.hif_setup(dim, n, m, a, w.dt, H.default_options(eps=0.0))
    x = np.random.default_rng(1).standard_normal(w.N)
    y = H.hif_apply(h, torch.from_numpy(A @ x).cuda()).cpu().numpy()
    assert np.linalg.norm(y - x) <= 1e-9 * np.linalg.norm(x)
    level0 = read_blob(H.hif_export_factor(h))["levels_data"][0][0]
    for cell in level0[:2] + level0[-1:]:
        I, B, G, V = cell
        AII = A[I][:, I].toarray()
        Ginv = np.linalg.inv(np.linalg.cholesky(AII))
        assert np.linalg.norm(G - Ginv) <= 1e-11 * np.linalg.norm(Ginv)
        Vref = np.linalg.solve(AII, A[I][:, B].toarray()).T
        assert np.linalg.norm(V - Vref) <= 1e-11 * np.linalg.norm(Vref)
    h.close()
