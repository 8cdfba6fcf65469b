"""Rules of the CTA-pair product kernel that can be read off its source (no GPU)."""
import os
import re

from paper_2608_25469_gb300 import build

KERNEL = os.path.join(build.CSRC, "tc_gemm.cuh")


def _block(text, start):
    """The brace-delimited block that opens at or after `start`."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def _kernel():
    text = re.sub(r"//[^\n]*", "", open(KERNEL).read())
    return _block(text, text.index("tc_gemm_kernel("))


def test_both_ctas_wait_for_every_commit_they_receive():
    """tc_commit_pair arrives on the barrier of both CTAs of the pair: each of them has to wait for
    its own, or it can leave with an arrival outstanding.  So every such barrier has a wait outside
    the code that only the first CTA runs."""
    body = _kernel()
    first_only = [_block(body, m.end()) for m in re.finditer(r"if \(rank == 0\) (?=\{)", body)]
    assert first_only
    both = body
    for b in first_only:
        both = both.replace(b, "")
    for bar in set(re.findall(r"tc_commit_pair\(&(\w+)", body)):
        assert re.search(r"mbar_wait\w*\(&%s\b" % bar, both), bar
