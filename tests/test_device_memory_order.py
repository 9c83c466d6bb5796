"""Promises about memory order that the kernels' sources make and no run can be relied on to break."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_26300_b200", "csrc")


def code(name):
    """A source file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", f.read(), flags=re.S))


def test_completion_word_is_stored_behind_what_the_counter_showed():
    """The last CTA of a host-buffer step learns from a counter that the others' results are on their way.  Every CTA fences
    its own results before it counts itself; the last one fences at system scope between the count and the word."""
    src = code("ckv_unitstep.cu")
    count, store = src.index("atomicAdd(done.ctas"), src.index("(volatile int *)done.flag = ")
    assert "__threadfence" in src[:count].rsplit("__syncthreads()", 1)[1]
    assert "__threadfence_system()" in src[count:store]
