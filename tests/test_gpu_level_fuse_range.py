"""Which levels of the FP32 apply run as fused launches, and through what a handle keeps them.

A level's cells leave the fused range when they are whole and go to the S-form
kernels: 608 cells and more, or cells of at most 32 rows.  From there up to the root
every level is fused in these factors, one launch a level and direction; CTAs of 256
threads above 16 parent cells (64 and 256 here), of 512 from 16 down.

Bars: exactly the expected launches, once each; after hif_refactor the bits of a
fresh handle, after hif_offload and hif_reload the bits of before.
"""

import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# dim, n, leaf, eps, lowest fused entity level
CASES = [(2, 8, 4, 1e-6, 0), (2, 8, 2, 1e-6, 1), (2, 36, 9, 0.5, 1), (2, 64, 8, 1e-6, 0), (2, 128, 4, 1e-3, 0),
         (2, 132, 33, 1e-6, 0), (2, 320, 10, 1e-3, 0), (2, 704, 11, 1e-3, 1), (3, 8, 4, 1e-4, 0), (3, 12, 3, 1e-2, 0)]


def _handle(case, seed=12):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_05566_gb300.hifcn as H
    dim, n, m, eps, _ = case
    w = W.small_variable_2d(n=n, m=m, dim=dim, eps=eps, contrast=1e2, dt=0.1, seed=seed)
    a = torch.from_numpy(w.a_nodes).cuda()
    h = H.hif_setup(dim, n, m, a, w.dt, H.default_options(eps=eps, precision=H.HIF_FP32))
    x = torch.randn(w.N, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    return H, h, a, x


def _apply(H, h, x):
    H.hif_stats_enable(h, True)
    y = H.hif_apply(h, x, precision=H.HIF_FP32)
    names = {r["name"]: r["launches"] for r in H.hif_stats_read(h) if r["name"].startswith("level_")}
    H.hif_stats_enable(h, False)
    return y, names


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}d_n{c[1]}_m{c[2]}" for c in CASES])
def test_fused_launches(case):
    dim, n, m, eps, first = case
    H, h, _, x = _handle(case)
    L = (n // m).bit_length() - 1
    want = {"level_top": 1}
    for l in range(first, L - 1):
        want[f"level_fwd_l{l}"] = want[f"level_bwd_l{l}"] = 1
    assert _apply(H, h, x)[1] == want
    h.close()


@pytest.mark.parametrize("case", [CASES[4], CASES[7]], ids=["n128", "n704"])
def test_handle_keeps_its_fused_levels(case):
    import torch
    H, h, a, x = _handle(case)
    y, names = _apply(H, h, x)
    H.hif_offload(h)
    H.hif_reload(h)
    y1, names1 = _apply(H, h, x)
    assert torch.equal(y1, y) and names1 == names
    _, f, a2, _ = _handle(case, seed=13)
    H.hif_refactor(h, a2)
    y2, names2 = _apply(H, h, x)
    assert torch.equal(y2, _apply(H, f, x)[0]) and names2 == names
    h.close()
    f.close()
