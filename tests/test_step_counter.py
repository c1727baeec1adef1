"""CPU checks of the device step counter's protocol in the sources: every block of a step's last launch
is counted, also one whose bounded wait ran out, and a new call starts from a count of zero.  A
block that leaves uncounted would let a later step's count fill up early: the step number then
advances while blocks still run, and a checkpoint lands one slot too far."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_13379_gb300", "csrc")


def _block(text, start):
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]


def _kernel(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "nf_mf.cu")).read())
    return _block(text, re.search(r"\n(?:__global__ void )?" + name + r"\(", text).start())


def test_a_block_that_gives_up_is_counted():
    body = _kernel("mf_pair_packed_kernel")
    gave_up = _block(body, body.index("if (timed_out)"))
    assert "return" in gave_up and re.search(r"MODE == 1\)[^;]*step_done\(", gave_up)
    # every other way out of the kernel is its end, where MODE 1 counts the block too
    assert body.count("return") - len(re.findall(r"\[&\]", body)) <= gave_up.count("return")
    assert len(re.findall(r"step_done\(", body)) == 2


def test_a_new_call_starts_the_count_at_zero():
    assert re.search(r"\*done_ctr\s*=\s*0", _kernel("set_clock_kernel"))
