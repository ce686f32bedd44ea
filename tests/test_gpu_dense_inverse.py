"""Batched inverse factors at the edges of the doubling.

The inverse of a Cholesky factor goes by block columns up to 256 rows and by
doubling (32, 64, ...) above.  Checked on the root and the cells of exact factors,
the root with 253, 257, 261 and 509 DOFs in 2D around and above the rule, and with
631 and 1261 in 3D (partial last blocks).

Bar: A = I - theta dt M applied to the exact inverse gives the vector back within
1e-9 (A >= I, ||A|| < 1e6, FP64 rounding).
"""

import numpy as np
import pytest

import workloads as W
from oracle import grid

pytestmark = pytest.mark.gpu

# dim, n, leaf: root 2 (n - 1) - 1 = 253, 257, 261 and 509 in 2D
CASES = [(2, 128, 64), (2, 130, 65), (2, 132, 33), (2, 256, 64), (3, 16, 8), (3, 22, 11)]


@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_n{n}_m{m}" for d, n, m in CASES])
def test_inverse_factors(case):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=0.0, contrast=1e2, dt=0.2, seed=2)
    h = H.hif_setup(dim, n, m, torch.from_numpy(w.a_nodes).cuda(), w.dt, H.default_options(eps=0.0))
    size = 2 * (n - 1) - 1 if dim == 2 else 3 * (n - 1) ** 2 - 3 * (n - 1) + 1
    assert H.hif_query(h)["root_size"] == size
    x = np.random.default_rng(5).standard_normal(w.N)
    b = grid.assemble_A(w.a_nodes, w.dt) @ x
    y = H.hif_apply(h, torch.from_numpy(b).cuda()).cpu().numpy()
    assert np.linalg.norm(y - x) <= 1e-9 * np.linalg.norm(x)
    h.close()
