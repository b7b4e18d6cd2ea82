"""What the kernels that issue MMAs and copies wait for before they free their tensor memory, read from their source.
A wait may give up in any warp, the issuing one or another: so the issuing warp waits (bounded) for its last MMAs on
every way out, not only when its own wait was the one that failed."""
import re

import pytest

from test_wait_agreement import body, code


def enclosing(text, at):
    """Headers of the blocks around text[at], outermost first."""
    stack, start = [], 0
    for k in range(at):
        c = text[k]
        if c == "{":
            stack.append(text[start:k].strip())
            start = k + 1
        elif c == "}":
            stack.pop()
            start = k + 1
        elif c == ";":
            start = k + 1
    return stack


# the wait for the last MMAs a warp issued
DRAINS = [("gram_high_tc.cu", "gram_rbf_high_tc_kernel", r"mbar_wait_bounded\(&mma_done\[\(issued - 1\) & 1\]"),
          ("gram_rbf_tc.cu", "gram_rbf_tc_sym_kernel", r"mbar_wait_bounded\(&mma_done\[\(q - 1\) % kSymBufs\]"),
          ("gram_rbf_tc.cu", "gram_rbf_tc_multi_kernel", r"mbar_wait_bounded\(&mma_done\[\(q - 1\) & 1\]"),
          ("batch.cu", "batch_kv_tmem_kernel", r"dwait\(&drain\[0\]"),
          ("batch.cu", "batch_kv_tmem_kernel", r"dwait\(&drain\[1\]"),
          ("batch.cu", "batch_kv_kernel", r"dwait\(drain")]


@pytest.mark.parametrize("name,kernel,wait", DRAINS)
def test_the_last_mmas_are_waited_for_on_every_way_out(name, kernel, wait):
    b = body(code(name), kernel)
    m = list(re.finditer(wait, b))
    assert len(m) == 1
    blocks = enclosing(b, m[0].start())
    assert not any("ok" in h for h in blocks), blocks
    assert not any(h.startswith(("for", "while")) for h in blocks), blocks
