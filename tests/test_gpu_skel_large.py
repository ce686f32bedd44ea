"""Skeletonization of entities above 64 DOFs (kernels spread over the chip).

Faces of 81, 121 and 225 DOFs (3D) and edges of 65 (2D), at tolerances that keep
everything (eps = 0), most, and almost nothing, against the oracle.  Bars, as
for the setup everywhere: the CN solution within 1e-9 at CG tolerance 1e-10 and
the iteration count within 1 (several factors are valid, their quality is not);
at eps = 0 one iteration; F^{-1} symmetric to 1e-11.
"""

import numpy as np
import pytest

import workloads as W
from parity import rel_err
from oracle import grid, hif, pcg

pytestmark = pytest.mark.gpu

CASES = [(3, 20, 10, 0.0), (3, 20, 10, 1e-4), (3, 20, 10, 0.5), (3, 24, 12, 1e-6), (3, 32, 8, 1e-3),
         (2, 132, 66, 1e-6)]


@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_n{n}_m{m}_eps{e:g}" for d, n, m, e in CASES])
def test_large_entities(case):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m, eps = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=eps, contrast=1e2, dt=0.1, seed=17)
    F = hif.factor(grid.assemble_A(w.a_nodes, w.dt), n, dim, m, eps)
    ref, it_ref, _ = pcg.cn_solve(w.a_nodes, w.u0, w.dt, 1, m, eps, (1, 1.0, 1.0), tol=1e-10, factor=F)
    h = H.hif_setup(dim, n, m, torch.from_numpy(w.a_nodes).cuda(), w.dt,
                    H.default_options(eps=eps, cg_tol=1e-10))
    H.hif_set_reaction(h, 1, 1.0, 1.0)
    u1, it = H.cn_step(h, torch.from_numpy(w.u0.ravel().copy()).cuda())
    assert rel_err(u1.cpu().numpy(), ref.ravel()) <= 1e-9
    assert abs(it - it_ref[0]) <= 1
    if eps == 0.0:
        assert it == 1
    rng = np.random.default_rng(4)
    x, y = (torch.from_numpy(rng.standard_normal(w.N)).cuda() for _ in range(2))
    fx, fy = H.hif_apply(h, x), H.hif_apply(h, y)
    assert abs(float(fx @ y - x @ fy)) <= 1e-11 * float(fx.norm() * y.norm())
    h.close()
