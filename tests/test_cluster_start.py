"""Kernels that write into other CTAs' shared memory wait for the whole cluster to have started first: a cluster
barrier on every path before the first round.  A missing one is a race that no run shows reliably, so this reads the
source."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_13804_gb300", "csrc")


def _top_level(source, kernel, until):
    """The kernel's statements outside any inner braces, up to `until`."""
    text = re.sub(r"//[^\n]*", "", source)
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
    with open(os.path.join(CSRC, name)) as f:
        source = f.read()
    statements = _top_level(source, kernel, "while (nsel < k_max)")
    assert re.search(r"(^|;|\})\s*cluster\.sync\(\);", statements), "a CTA may write to a peer that has not started"
