"""Merged batched steps in which a CTA meets the cells of handles that are done.

The S-form cells of all handles go through one launch, a few cells a CTA; those of
a handle whose solve has ended are passed over.  HIFCN_TMA_GRID holds the launch
at one to five CTAs, so that every CTA passes from working cells to idle ones and
back: zero right-hand sides first, between and last, loose factors that need
several iterations beside tight ones, 2D and 3D.

Bars: each state equals its single step within 1e-9 (CG tolerance 1e-10), counts
within 1, idle handles stay at zero.
"""

import pytest

import workloads as W
from parity import rel_err

pytestmark = pytest.mark.gpu

# dim, n, leaf, eps, zero state
SPEC = [(2, 32, 4, 1e-6, 1), (2, 64, 8, 1e-2, 0), (2, 64, 8, 1e-6, 1), (2, 32, 16, 1e-6, 0), (3, 16, 4, 1e-4, 1),
        (3, 16, 4, 1e-2, 0), (2, 64, 4, 1e-6, 0), (2, 36, 9, 1e-6, 1)]


@pytest.mark.parametrize("cap", ["1", "2", "5"])
def test_idle_handles_between_working_ones(cap, monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    hs, us = [], []
    for i, (dim, n, m, eps, zero) in enumerate(SPEC):
        w = W.small_variable_2d(n=n, m=m, dim=dim, eps=eps, contrast=1e2, dt=0.2, seed=50 + i)
        h = H.hif_setup(dim, n, m, torch.from_numpy(w.a_nodes).cuda(), w.dt,
                        H.default_options(eps=eps, precision=H.HIF_FP32, cg_tol=1e-10))
        H.hif_set_reaction(h, 1, 1.0, 1.0)
        hs.append(h)
        us.append(torch.from_numpy(w.u0.ravel().copy() * (0.0 if zero else 1.0)).cuda())
    single = [H.cn_step(h, u) for h, u in zip(hs, us)]
    assert len({it for _, it in single}) > 2  # none, few and several iterations
    monkeypatch.setenv("HIFCN_TMA_GRID", cap)
    outs, its = H.cn_step_batched(hs, us)
    for i, (ref, it) in enumerate(single):
        if SPEC[i][4]:
            assert its[i] == 0 and float(outs[i].abs().max()) == 0.0
            continue
        assert rel_err(outs[i].cpu().numpy(), ref.cpu().numpy()) <= 1e-9, i
        assert abs(its[i] - it) <= 1, (i, its[i], it)
    for h in hs:
        h.close()
