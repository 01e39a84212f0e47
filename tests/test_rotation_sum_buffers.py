"""The buffers of the conjugate-gradient kernel's grid-wide sums, read from its source: a block may write a
buffer that other blocks read only with a grid barrier behind those reads, and may read it only with one
behind the writes. (Nothing orders the blocks but the barrier, so a missing one shows up on a GPU only by
chance: in the wrong sum of a block that came late.) The statements are taken in the order of the text,
the body of the iterations twice."""
import os
import re

import pytest

from paper_2605_18052_gb300 import build

EVENT = re.compile(r"(?P<write>\w+)\[(?:kb / RT_CAMS|kc)\] =|sum_values\((?P<read>\w+)|(?P<barrier>gb\.wait\(\))")


def _kernel():
    text = open(os.path.join(build.CSRC, "fm_rotation.cu")).read()
    text = re.sub(r"//[^\n]*", "", text)
    body = text[text.index("k_cg_solve(DevRot t"):text.index("gb.finish();")]
    at = body.index("for (int c = 0; c < CG_CHUNK; ++c)")
    return body[:at], body[at:]


def _violations(setup, loop):
    written, read, bad = set(), set(), []      # buffers touched since the last barrier
    for m in list(EVENT.finditer(setup)) + 2 * list(EVENT.finditer(loop)):
        if m["barrier"]:
            written, read = set(), set()
        elif m["write"]:
            bad += [m["write"]] if m["write"] in read else []
            written.add(m["write"])
        else:
            bad += [m["read"]] if m["read"] in written else []
            read.add(m["read"])
    return bad


def test_no_sum_is_overwritten_while_another_block_reads_it():
    setup, loop = _kernel()
    assert {m["write"] for m in EVENT.finditer(loop)} >= {"slot", "cam_rz"}   # the pattern finds the sums
    assert _violations(setup, loop) == []


@pytest.mark.parametrize("old, new", [("slot_setup", "slot"), ("gb.wait()", "true")])
def test_the_check_sees_a_shared_buffer_and_a_missing_barrier(old, new):
    setup, loop = _kernel()
    assert _violations(setup.replace(old, new), loop.replace(old, new))
