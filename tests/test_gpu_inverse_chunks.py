"""A cell's inverse factor does not depend on the cells eliminated beside it.

G = L^{-1} goes by block columns for interiors of at most 256 DOFs and by doubling
above.  The level above the leaves of these factors has interiors on both sides of
256, so a rule on the largest cell of a chunk would sum the smaller ones in another
order when they are eliminated one by one.

Bar: the exported factors are equal byte for byte.
"""

import pytest

import workloads as W
from blobutil import read_blob

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [17, 18])
def test_chunks_on_both_sides_of_the_rule(seed, monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m, eps = 3, 24, 6, 0.025
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=eps, contrast=1e4, dt=0.1, seed=seed)
    a = torch.from_numpy(w.a_nodes).cuda()

    def blob():
        h = H.hif_setup(dim, n, m, a, w.dt, H.default_options(eps=eps))
        out = H.hif_export_factor(h)
        h.close()
        return out

    ref = blob()
    sizes = [len(c[0]) for c in read_blob(ref)["levels_data"][1][0]]
    assert min(sizes) <= 256 < max(sizes), sizes
    monkeypatch.setenv("HIFCN_SETUP_FRONT_BYTES", "65536")
    assert blob() == ref
