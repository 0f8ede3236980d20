"""The convolution kernels' time-out paths wait for every copy they armed a barrier for, so that no
copy still aims at shared memory that the next block may own.  A wait that runs out cannot be made
to happen without harm, so the sources are read as text."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = re.sub(r"//[^\n]*", "", open(os.path.join(ROOT, "paper_2412_03451_gb300", "csrc", "ps_conv.cu")).read())


def body(kernel):
    m = re.search(r"__global__[^;{]*\b%s\([^{;]*\)\s*\{" % kernel, SRC)
    depth, i = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(SRC[i], 0)
        i += 1
    return SRC[m.end():i]


def armed(text):
    """Barriers that copies are armed for: names, without indices and address conversions."""
    return {re.sub(r"^smem_u32\(&|\[.*", "", x) for x in re.findall(r"mbar_expect\(([\w&(]+(?:\[\w+\])?)", text)}


@pytest.mark.parametrize("kernel, flag, barriers", [("k_conv_first", r"if \(!ok\) \{", {"bw", "bp"}),
                                                    ("k_conv_inner", r"if \(\(failed \|\| out_failed\)", {"w_full", "f"}),
                                                    ("k_wgrad", r"if \(failed", {"f"})])
def test_time_out_waits_for_every_armed_barrier(kernel, flag, barriers):
    text = body(kernel)
    aliases = {"full": "f"}
    assert {aliases.get(b, b) for b in armed(text)} == barriers
    drain = text[[m.start() for m in re.finditer(flag, text)][-1]:]
    for b in barriers:
        assert re.search(r"mbar_wait\((?:smem_u32\(&)?%s\b" % {"f": "full"}.get(b, b), drain), b


def test_no_patch_is_loaded_after_a_failed_wait():
    text = body("k_conv_first")
    # the loop is not entered unless every thread saw the weights, and a load is counted
    # whether or not the wait for it runs out
    assert re.search(r"ok = !__syncthreads_or\(!mbar_wait\(bw, 0\)\);", text)
    assert re.search(r"for \([^;]*; ok && [^;]*;", text)
    assert "ok = mbar_wait(bp, np++ & 1);" in text
