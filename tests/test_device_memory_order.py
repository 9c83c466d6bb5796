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


def test_words_of_any_content_are_subtracted_as_unsigned_numbers():
    """The selection compares by the sign of a difference, also for words past the unit's scores, which hold what the ring left
    (negative numbers among them) and whose bits are masked: as signed numbers that would overflow."""
    src = code("ckv_unitstep.cu")
    assert src.count("- key[j][e]") == 2 and "(int)key[j][e]" not in src
    assert re.search(r"const uint32_t lo1 = ", src) and re.search(r"const uint32_t hi1 = ", src)


def test_barriers_are_set_up_before_other_lanes_of_the_producer_warp_use_them():
    """One lane initialises the ring's barriers, its neighbours issue fills on them, and no barrier that waits lies between the
    two: the warp is synchronised right behind the initialisation."""
    src = code("ckv_unitstep.cu")
    init = src.index("fence_barrier_init()")
    assert init < src.index("if (warp == kProducerWarp) __syncwarp()", init) < src.index("cluster_arrive_release()", init)
    assert src.index("cluster_arrive_release()", init) < src.index("fill_tile(lane, lane", init)


def test_kernels_that_start_early_do_not_call_their_inputs_constant():
    """A programmatic dependent launch runs while the launch ahead of it still writes: `__ldg` and `const __restrict__`
    would let the compiler move loads up past griddepcontrol.wait."""
    kernels = re.compile(r"ckv_launch_pdl\(\s*\(?(\w+)")
    early = {"ckv_attn_mma.cu", "ckv_scan.cu", "ckv_select.cu", "ckv_stats.cu", "ckv_unitstep.cu"}
    found = {f for f in os.listdir(CSRC) if f.endswith(".cu") and (kernels.search(code(f)) or "griddepcontrol" in code(f)
                                                                    or "cudaLaunchAttributeProgrammatic" in code(f))}
    assert found == early   # a new one belongs into the list
    for name in sorted(early | {"ckv_blockstats.cuh", "ckv_scanpart.cuh", "ckv_attnpage.cuh"}):
        src = code(name)
        src = re.sub(r"__global__[^;{]*ckv_stats_export_kernel.*?\n}\n", "", src, flags=re.S)   # an ordinary launch
        for bad in (r"__ldg", r"ld\.global\.nc", r"load8<true>", r"load8<NC>", r"load_split8\(", r"const\s+[\w ]+\*\s*__restrict__"):
            assert not re.search(bad, src), (name, bad)
