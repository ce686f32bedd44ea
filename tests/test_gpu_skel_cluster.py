"""The pivoted QR of large entities does not depend on the cluster it runs in.

Entities of 81 to 225 DOFs, all of a sub-step in one launch (clusters of one to a
few CTAs, more clusters than fit the chip at once) and one entity a launch
(scratch limit; clusters of 16).  Every column norm is summed by one warp and ties
go to the smaller column, so the exported factors are equal byte for byte, and so
are those of repeated setups.
"""

import pytest

import workloads as W

pytestmark = pytest.mark.gpu

CASES = [(3, 20, 10, 1e-4), (3, 40, 10, 1e-3), (3, 32, 8, 1e-3), (2, 132, 66, 1e-6)]


@pytest.mark.parametrize("case", CASES, ids=[f"{d}d_n{n}_m{m}" for d, n, m, _ in CASES])
def test_factor_does_not_depend_on_the_cluster(case, monkeypatch):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m, eps = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=eps, contrast=1e2, dt=0.1, seed=23)
    a = torch.from_numpy(w.a_nodes).cuda()

    def blob():
        h = H.hif_setup(dim, n, m, a, w.dt, H.default_options(eps=eps))
        out = H.hif_export_factor(h)
        h.close()
        return out

    ref = blob()
    for _ in range(2):
        assert blob() == ref
    monkeypatch.setenv("HIFCN_SETUP_SCRATCH_BYTES", "65536")
    assert blob() == ref
