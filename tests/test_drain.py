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


# Kernels that double-buffer column tiles: thread 0 leaves after a wait that gave up only once the copies it has issued
# have landed: one column tile before the loop, tiles 0 .. q + 1 at the wait for tile q.
TILE_KERNELS = [("gram_f32.cu", "gram_f32_kernel"), ("gram_f32_sym.cu", "gram_f32_sym_kernel"),
                ("gram_high.cu", "gram_lap_high_kernel"), ("gram_high.cu", "gram_rbf_emu_kernel"),
                ("gram_high_sym.cu", "gram_lap_high_sym_kernel")]


@pytest.mark.parametrize("name,kernel", TILE_KERNELS)
def test_tile_kernels_drain_before_they_leave(name, kernel):
    b = body(code(name), kernel)
    waits = [m.start() for m in re.finditer(r"\bmbar_wait_bounded\(", b)]
    assert len(waits) == 2 and len(re.findall(r"\breturn\b", b)) == 2
    for w, issued in zip(waits, (r"(?:1|min\(jt1 - jt0, 1\))", r"min\(q \+ 2, jt1 - jt0\)")):
        assert re.match(r"mbar_wait_bounded\([^;{]*\) \{\s*if \(tid == 0\) tile_drain\(bars, " + issued +
                        r", err\);\s*return;\s*\}", b[w:]), b[w:w + 200]


def test_plain_tensor_core_kernel_drains_on_abort():
    b = body(code("gram_rbf_tc.cu"), "gram_rbf_tc_kernel")
    abort = b[b.index("if (*abort_flag) {"):]
    abort = abort[:abort.index("break;")]
    assert "tile_drain(bars, min(nt, max(2, q + 1)), err);" in abort and "mma_drain(bars + 3, max(0, q - 1), min(q + 1, nt), err);" in abort
