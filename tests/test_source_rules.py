"""Rules of memory order that no run can show to hold, checked on the sources."""
import os
import re

from native import HERE

CSRC = os.path.join(os.path.dirname(HERE), "paper_2412_20105_b200", "csrc")


def _code(name):
    """The source without comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def _body(src, head):
    """The braces' contents of the definition that starts with `head`."""
    i = src.index("{", src.index(head))
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        j += 1
    return src[i:j]


def test_rows_behind_a_flag_are_fenced_between_the_proxies():
    """The selection moves rows with ordinary stores, the attention reads them with bulk copies: a proxy fence on both
    sides of the flag, and no look-up of a flag around it."""
    attend, finish = _code("st3_attend.cuh"), _code("st3_finish.cuh")
    seen = _body(attend, "bool flag_seen(")
    assert seen.index("ld_acquire(") < seen.index("proxy_fence()")
    assert attend.count("ld_acquire(") == 2                       # its definition and flag_seen
    moves = finish[finish.index("kMoveBatch = 8"):]
    assert moves.index("proxy_fence()") < moves.index("done()")
    assert "fence.proxy.async" in _body(_code("st3_common.cuh"), "void proxy_fence(")


def test_launches_that_start_early_read_inputs_with_ordinary_loads():
    """A read-only load may be moved above griddepcontrol.wait and promises that nobody writes while the kernel runs;
    the launch ahead of one that starts early may.  What was complete before the grid can start is exempt: the text
    lengths, and the prompt where the kept rows are copied."""
    attend, st3, prefill = _code("st3_attend.cuh"), _code("st3.cu"), _code("st3_prefill.cu")
    assert re.findall(r"__ldg\(([^)]*)\)", attend) == ["p.text_len + b"]
    assert "__restrict__" not in attend + _code("st3_finish.cuh") + prefill and "__ldg" not in prefill
    cluster = st3[st3.index("st3_na_cluster_kernel("):]
    assert "__restrict__" not in cluster[:cluster.index("{")]
    assert "__ldg" not in _body(st3, "st3_na_cluster_kernel(")
    gather = _body(_code("st3_finish.cuh"), "st3_gather_kernel(")
    assert set(re.findall(r"__ldg\((\w+)", gather)) == {"p", "srcK", "srcV"}


def test_limits_on_waits_do_not_count_the_work_ahead():
    """In a launch that starts early a limit runs only once the launch ahead has ended: the attention kernel restarts its
    clock until a manager has waited for that launch, the prompt attention waits for it first."""
    attend = _code("st3_attend.cuh")
    wait = _body(attend, "bool ring_wait(")
    assert wait.index("if (abort_flag[1])") < wait.index("else if (clock64() - t0 > kWaitCycles)")
    assert "s_abort[1] = p.order;" in attend
    waits = [m.end() for m in re.finditer("griddepcontrol.wait", attend)]
    assert len(waits) == 3 and all("abort_flag[1] = 0;" in attend[i:i + 200] for i in waits[:2])    # and one at the end
    prompt = _body(_code("st3_prefill.cu"), "st3_prefill_attend_kernel(")
    assert prompt.index("griddepcontrol.wait") < prompt.index("__syncthreads()") < prompt.index("pf_wait")


def test_tensor_memory_is_taken_before_a_successor_may_start():
    """A successor that takes all tensor memory of an SM ahead of its own wait would otherwise keep a block of the prompt
    attention from its share, and wait for that block."""
    prompt = _body(_code("st3_prefill.cu"), "st3_prefill_attend_kernel(")
    alloc = prompt.index("tcgen05.alloc")
    assert alloc < prompt.index("__syncthreads()", alloc) < prompt.index("griddepcontrol.launch_dependents")


def test_a_block_that_gives_up_waits_for_its_copies():
    attend = _code("st3_attend.cuh")
    left = attend[attend.index("publish(slot0, po);"):attend.index("s_desc[s].info = -1;")]
    assert "if (cur_valid) {" in left and left.count("copy_settled(") == 2 and "bulk_written()" in left
    settled = _body(attend, "bool copy_settled(")
    assert "kWaitCycles" in settled and "abort" not in settled
