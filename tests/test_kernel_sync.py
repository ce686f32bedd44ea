"""Synchronisation that a passing run cannot show, read from the kernels' source.

A missing barrier seldom changes a result, and provoking one on a GPU is no
test; the order of the statements is checked instead.
"""

import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2004_05566_gb300" / "csrc"


def _body(file, name):
    """Text of function `name` of a source file, comments removed."""
    text = re.sub(r"//[^\n]*", "", (CSRC / file).read_text())
    at = re.search(r"\b%s\([^;{]*\)\s*\{" % name, text)
    depth, i = 1, at.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[at.end():i]


def test_cluster_has_started_before_its_shared_memory_is_written():
    body = _body("setup.cu", "k_skel_qr")
    assert 0 <= body.find("cluster_sync();") < body.find("cluster_store(")
    # and none of its CTAs leaves while another may still store
    assert body.rfind("cluster_sync();") > body.rfind("cluster_store(")


def test_scalars_of_a_panel_step_are_read_before_the_next_are_written():
    body = _body("dense_batched.cuh", "k_chol_diag")
    loop = body[body.index("for (int k = 0; k < jb; ++k)"):]
    # one warp writes and reads s_r; its reads after the last CTA barrier of a step
    # end at a warp barrier
    tail = loop[loop.index("if (q == 0)", loop.rindex("D[i][j] -=")):]
    read = max(tail.index("s_r[0]"), tail.index("s_r[2]"))
    assert "__syncwarp();" in tail[read:tail.index("A[(j0 + i)")].split("__syncthreads();")[0]


def test_copy_warp_releases_the_cell_buffer():
    # cm[b] is read by the consumers and by the copy warp: the gather warp refills it
    # after both have arrived
    for kernel in ("k_cell_fwd_tma_S", "k_cell_bwd_tma_S"):
        body = _body("apply.cu", kernel)
        assert re.search(r"mbar_init\(&freed\[b\], kConsumerWarps \+ 1\);", body)
        assert re.search(r"produce_cells<[^;]*\bfreed\b[^;]*;", body)
    body = _body("apply.cu", "produce_cells")
    chunks = body[body.index("for (int j = 0; j < nch"):]
    assert chunks.index("mbar_arrive(&freed[bb]);") > chunks.index("bulk_load(")
    assert "cm[" not in chunks
