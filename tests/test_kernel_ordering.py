"""Ordering rules of the CUDA sources whose violation no run on a GPU shows reliably
(a race between lanes, a cached load), checked on the source text."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_01086_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _body(src, head):
    """Text of the brace block that follows the first match of `head`."""
    at = src.index("{", re.search(head, src).end())
    depth = 0
    for i in range(at, len(src)):
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        if depth == 0:
            return src[at:i + 1]
    raise AssertionError(head)


def test_levels_are_rewritten_behind_a_barrier():
    """stream_tiles moves the symbols left over the levels that the lanes of a step
    read: a warp barrier lies between the last step and the first of those stores."""
    body = _body(_source("warp_tile.cuh"), r"void stream_tiles\(")
    after = body[body.rindex("step(sg, dd,"):]
    first_store = min(m.start() for m in re.finditer(r"stage\s*\+\s*at\)\s*=[^=]|stage\[at\]\s*=[^=]", after))
    assert "__syncwarp()" in after[:first_store]


def test_levels_of_overlapped_encoder_kernels_are_plain_loads():
    """k_enc_starts, k_enc_scan and k_enc_pack may start while the level kernels
    still write: what they read through the read-only path is the code table and
    nothing else."""
    src = _source("encode.cu")
    table = re.compile(r"__ldg\((p\.code_tab|gt|tab)\b")
    for head in (r"uint4 load_run16\(", r"k_enc_starts\(", r"void walk_block\(", r"k_enc_scan\(", r"k_enc_pack\("):
        body = _body(src, head)
        assert len(re.findall(r"__ldg\(", body)) == len(table.findall(body)), head
