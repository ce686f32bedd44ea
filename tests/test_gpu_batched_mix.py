"""Merged batched steps over levels of both kinds.

S-form levels of all handles go through one bulk-copy launch, the others through
one CTA per cell, in the same phase: leaf interiors of 9, 49, 256 (S-form) and 289
DOFs (not), 3D cells, one to four levels, a handle whose right-hand side is zero
(inactive from the start) and handles that need different iteration counts
(eps 1e-6 and 1e-2), and a true-residual period that falls due.

Bars: each state equals its single step within 1e-9 (CG tolerance 1e-10), counts
within 1; a handle's bits do not depend on the batch.
"""

import numpy as np
import pytest

import workloads as W
from parity import rel_err

pytestmark = pytest.mark.gpu

# dim, n, leaf, eps, zero state, true-residual period
SPEC = [(2, 32, 4, 1e-6, 0, 50), (2, 64, 8, 1e-2, 0, 2), (2, 68, 17, 1e-6, 0, 50), (2, 36, 18, 1e-6, 0, 1),
        (3, 16, 4, 1e-4, 0, 50), (2, 64, 8, 1e-6, 1, 50), (2, 8, 4, 1e-6, 0, 3)]


def test_merged_mix():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    hs, us = [], []
    for i, (dim, n, m, eps, zero, period) in enumerate(SPEC):
        w = W.small_variable_2d(n=n, m=m, dim=dim, eps=eps, contrast=1e2, dt=0.2, seed=30 + i)
        h = H.hif_setup(dim, n, m, torch.from_numpy(w.a_nodes).cuda(), w.dt,
                        H.default_options(eps=eps, precision=H.HIF_FP32, cg_tol=1e-10, true_res_period=period))
        H.hif_set_reaction(h, 1, 1.0, 1.0)
        hs.append(h)
        us.append(torch.from_numpy(w.u0.ravel().copy() * (0.0 if zero else 1.0)).cuda())
    outs, its = H.cn_step_batched(hs, us)
    for i, (h, u) in enumerate(zip(hs, us)):
        ref, it = H.cn_step(h, u)
        if SPEC[i][4]:
            assert its[i] == 0 and float(outs[i].abs().max()) == 0.0
            continue
        assert rel_err(outs[i].cpu().numpy(), ref.cpu().numpy()) <= 1e-9, i
        assert abs(its[i] - it) <= 1, (i, its[i], it)
    for i in (0, 3, 4):
        alone, _ = H.cn_step_batched([hs[i]], [us[i]])
        assert torch.equal(alone[0], outs[i])
    order = [4, 0, 6, 3, 2]
    mixed, _ = H.cn_step_batched([hs[i] for i in order], [us[i] for i in order])
    for k, i in enumerate(order):
        assert torch.equal(mixed[k], outs[i])
    for h in hs:
        h.close()
