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
