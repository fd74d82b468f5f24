"""Synchronisation that no run shows reliably when it is missing, read from the kernels' sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_13804_gb300", "csrc")


def _source(name):
    """A source file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _top_level(text, kernel, until):
    """The kernel's statements outside any inner braces, up to `until`."""
    text = text[re.search(r"\b%s\(const BatchDesc" % kernel, text).start():]
    text = text[text.index("{") + 1:]
    depth, out = 0, []
    for i, ch in enumerate(text):
        if depth == 0 and text.startswith(until, i):
            return "".join(out)
        if ch == "}":
            depth -= 1
        if depth == 0:
            out.append(ch)
        if ch == "{":
            depth += 1
    raise AssertionError("no round loop in " + kernel)


@pytest.mark.parametrize("name,kernel", [("select.cu", "select_kernel"), ("select_gram.cu", "select_gram_kernel")])
def test_cluster_barrier_before_the_first_round(name, kernel):
    """Kernels that write into other CTAs' shared memory wait for the whole cluster to have started first: a
    cluster barrier on every path before the first round."""
    statements = _top_level(_source(name), kernel, "while (nsel < k_max)")
    assert re.search(r"(^|;|\})\s*(cluster\.sync|cluster_sync_all)\(\);", statements), "a CTA may write to a peer that has not started"


def test_warp_waits_order_the_other_lanes():
    """A wait that lane 0 makes for its warp: a shuffle hands its outcome to the other lanes, but orders no memory;
    what they read afterwards is ordered by a __syncwarp()."""
    found = []
    for name in sorted(os.listdir(CSRC)):
        for m in re.finditer(r"SP_DEVINL bool (mbar_\w*_warp)\(.*?\n\}", _source(name), re.S):
            found.append(m.group(1))
            assert re.search(r"__syncwarp\(\);\s*return __shfl_sync\([^;]*;\s*\}$", m.group(0)), m.group(1)
    assert "mbar_wait_warp" in found and "mbar_poll_cluster_warp" in found
