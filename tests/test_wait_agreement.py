"""The bounded waits of the tensor-memory kernels, read from their source.  A wait can run out in some lanes of a
warp and not in others.  Loads from and stores to tensor memory are operations of the whole warp, so a warp that
does them takes the outcome of a wait by vote (__all_sync, or bwait_warp, which votes at every poll): a lane that
left alone would keep the others waiting for good, behind every bound."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_07929_gb300", "csrc")
WAIT = re.compile(r"\b(?:bwait|mbar_wait_bounded)\(")


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def body(text, kernel):
    at = text.index("{", text.index(")", re.search(r"\b" + kernel + r"\(", text).end()))
    # the parameter list holds no braces: the first one opens the body
    depth, k = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        k += 1
        if depth == 0:
            return text[at:k]


def call_at(text, at):
    """The text of the call whose name starts at `at`, to its closing parenthesis."""
    k = text.index("(", at)
    depth = 0
    while True:
        depth += {"(": 1, ")": -1}.get(text[k], 0)
        k += 1
        if depth == 0:
            return at, k


# (file, kernel, where the part of the warps that read tensor memory begins)
KERNELS = [("batch.cu", "batch_kv_kernel", r"const int lg = warp & 3"),
           ("batch.cu", "batch_kv_tmem_kernel", r"const int lq = warp & 3"),
           ("gram_rbf_tc.cu", "gram_rbf_tc_kernel", r"if \(q >= 1\) \{"),
           ("gram_rbf_tc.cu", "gram_rbf_tc_sym_kernel", r"const int lq = warp & 3"),
           ("gram_rbf_tc.cu", "gram_rbf_tc_multi_kernel", r"const int lq = warp & 3"),
           ("gram_high_tc.cu", "gram_rbf_high_tc_kernel", r"const int lq = warp & 3")]


@pytest.mark.parametrize("name,kernel,start", KERNELS)
def test_warps_that_read_tensor_memory_agree_on_their_waits(name, kernel, start):
    part = body(code(name), kernel)
    part = part[re.search(start, part).start():]
    votes = [call_at(part, m.start()) for m in re.finditer(r"\b__all_sync\(", part)]
    waits = [m.start() for m in WAIT.finditer(part)]
    assert waits or "bwait_warp(" in part
    for w in waits:
        assert any(a < w < b for a, b in votes), part[max(0, w - 120):w + 120]


def test_the_voting_wait_votes_on_every_answer():
    f = body(code("batch.cu"), "bwait_warp")
    assert re.search(r"if \(__all_sync\(0xffffffffu, mbar_try_wait\(bar, parity\)\)\) return true;", f)
    assert len(re.findall(r"return true;", f)) == 1
    assert re.search(r"__any_sync\(0xffffffffu, \*abort_flag\)\) return false;", f)
