"""Rules of the kernels' asynchronous copies, waits and barriers that no run
shows (a broken one corrupts memory or hangs only when the timing is bad),
checked on the kernels' source text."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_03275_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _block(text, start):
    """The brace block that begins at or after `start`: (first, last + 1)."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == "{") - (text[j] == "}")
        if depth == 0:
            return i, j + 1
    raise AssertionError("unbalanced braces")


def _kernel(text, name):
    start = text.index(f" {name}(")
    a, b = _block(text, start)
    return text[a:b]


def test_gptq_block_loop_leaves_no_copy_behind():
    """Leaving the block loop early waits for nothing, so every copy staged
    before that exit is under the condition that the exit is not taken."""
    k = _kernel(_source("gptq.cu"), "gptq_rows_kernel")
    end = k.index("if (!later) break;")
    calls = [m.start() for m in re.finditer(r"stage_u\(\w+, \d", k[:end])]
    assert calls
    guarded = [_block(k, m.end()) for m in re.finditer(r"if \(later\) (?=\{)", k[:end])]
    for c in calls:
        assert any(a < c < b for a, b in guarded), k[c:c + 20]


def test_barriers_behind_bounded_waits_are_reached_together():
    """A loop that leaves on its own bounded wait's outcome and has a barrier of
    several warps takes one outcome for all of them first: a warp that gave up
    alone would leave the others in the barrier for good."""
    seen = 0
    for name in sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")):
        text = _source(name)
        for m in re.finditer(r"\bfor \([^{;]*;[^{;]*;[^{;\n]*\) \{[ \t]*$", text, re.M):
            a, b = _block(text, m.end() - 1)
            body = text[a:b]
            bar, wait = body.find("named_bar_sync("), re.search(r"\b(mbar_wait|mbar_wait_warp|warp_wait)\(", body)
            if bar < 0 or not wait or wait.start() > bar:
                continue
            seen += 1
            assert "group_and(" in body[:bar], f"{name}: {m.group(0)}"
    assert seen


def test_copies_are_waited_for_before_a_thread_block_ends():
    """Whatever ends the loop of a warp that issues bulk copies (a bounded wait
    that ran out among it), the warp then waits for those in flight: each such
    warp's branch ends in waits on the barriers that its copies complete on."""
    seen = 0
    for name in ("decode.cu", "prefill.cu", "dense.cu"):
        text = _source(name)
        for m in re.finditer(r"\bif \(warp [^{]*\{", text):
            a, b = _block(text, m.end() - 1)
            body = text[a:b]
            loads = list(re.finditer(r"\b(?:tma_load_2d|tma_load_2d_pair|bulk_g2s|bulk_g2s_hint)_warp\(", body))
            if not loads:
                continue
            seen += 1
            last = list(re.finditer(r"\bmbar_wait_warp\(&\w*full\[", body))[-1].start()
            assert last > loads[-1].start(), f"{name}: {m.group(0)}"
    assert seen == 6


def test_mmas_are_waited_for_before_tensor_memory_is_freed():
    """The issuing warp's branch ends in a wait on a commit of all its MMAs."""
    seen = 0
    for name in ("decode.cu", "prefill.cu", "dense.cu"):
        text = _source(name)
        for m in re.finditer(r"\bif \(warp [^{]*\{", text):
            a, b = _block(text, m.end() - 1)
            body = text[a:b]
            mmas = list(re.finditer(r"\bumma_(?:bf16|bf16_ts|bf16_pair|mxf4_ts)_warp\(", body))
            if not mmas:
                continue
            seen += 1
            assert re.search(r"umma_commit(?:_pair)?_warp\(&(mma_done|acc_bar).*mbar_wait_warp\(&\1", body[mmas[-1].end():],
                             re.S), f"{name}: {m.group(0)}"
    assert seen == 6   # (the decode kernel: a branch within the branch)
