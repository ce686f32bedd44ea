"""HIFCN_ITEM_TARGET is taken literally, whatever its value.

512 3D leaf cells of 216 DOFs: left to itself the library cuts them finer than the
number of CTAs it aims at, by their bytes.  608 CTAs asked for by name are 608, as
607 and 609 are: the item lists of the three (16 bytes an item, part of the
handle's device bytes) have the same length, shorter than the automatic ones.
"""

import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_every_target_is_literal(monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m, eps = 3, 56, 7, 1e-2
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=eps, contrast=1e2, dt=0.1, seed=3)
    a = torch.from_numpy(w.a_nodes).cuda()

    def held():
        h = H.hif_setup(dim, n, m, a, w.dt, H.default_options(eps=eps, precision=H.HIF_FP32))
        out = H.hif_query(h)["device_bytes"]
        h.close()
        return out

    automatic = held()
    asked = {}
    for t in (607, 608, 609):
        monkeypatch.setenv("HIFCN_ITEM_TARGET", str(t))
        asked[t] = held()
    # ceil(t / cells) items a cell: the same for the three targets (512, 64 and 8 cells)
    assert asked[607] == asked[608] == asked[609], asked
    assert automatic > asked[608]
