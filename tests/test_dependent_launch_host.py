"""What cannot be tried on one GPU, or must not be, because getting it wrong is a wait without end or a race: the order of
the tensor-memory allocation, the dependency wait and the release of the dependents, read from the kernels' source.

A block that holds tensor memory while it waits for its predecessor is waited for by a predecessor on the same SM that
released its dependents before it allocated. So the default mode allocates behind the wait, an allocation ahead of it
needs a reason the host gives, and the kernel itself releases its dependents behind its own allocation."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_26577_b200", "csrc")


def _source(name="tree_attention_tc.cu"):
    text = re.sub(r"/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def _body(text, head):
    """The braces that follow `head`."""
    start = text.index("{", text.index(head))
    depth = 0
    for i in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start:i + 1]
    raise AssertionError("unbalanced braces")


def test_tensor_memory_is_taken_behind_the_wait():
    kernel = _body(_source(), "tree_attn_tc_kernel(const TcParams p")
    assert kernel.count("tcgen05.alloc") == 1
    take = _body(kernel, "auto tmem_take = [&]")
    assert "tcgen05.alloc" in take and take.index("tcgen05.alloc") < take.index("tcgen05.relinquish_alloc_permit")
    calls = [m.start() for m in re.finditer(r"\btmem_take\(\)", kernel)]
    guards = [re.search(r"if \((!?p\.tmem_first)\) $", kernel[:c]).group(1) for c in calls]
    assert guards == ["p.tmem_first", "!p.tmem_first"]
    default = _body(kernel, "if (!early)")
    order = [default.index(x) for x in ("griddepcontrol.wait", "tmem_take()", "griddepcontrol.launch_dependents")]
    assert order == sorted(order)


def test_dependents_are_released_by_the_warp_that_allocates():
    kernel = _body(_source(), "tree_attn_tc_kernel(const TcParams p")
    warp = re.search(r"if \(warp == (\d)\)", _body(kernel, "auto tmem_take = [&]")).group(1)
    released = [m.start() for m in re.finditer("griddepcontrol.launch_dependents", kernel)]
    assert len(released) == 2
    assert re.search(r"if \(warp == %s\) asm volatile\(\"$" % warp, kernel[:released[0]])
    early = kernel.rindex("if (warp == %s) {" % warp, 0, released[1])  # the producer's branch, which holds `if (early)`
    assert "griddepcontrol.wait" in kernel[early:released[1]] and released[1] < early + len(_body(kernel[early:], "if ("))


def test_a_launch_without_work_waits_for_its_predecessor():
    """What follows a launch waits for that launch alone: one that ended ahead of its predecessor would break the order of
    the stream. In the early mode a block without work leaves at once, so the first one waits on behalf of all."""
    kernel = _body(_source(), "tree_attn_tc_kernel(const TcParams p")
    idle = _body(kernel, "if (!wk.valid)")
    assert re.search(r"if \(early && blockIdx\.x == 0\) asm volatile\(\"griddepcontrol\.wait;", idle)
    assert idle.index("tmem_return()") < idle.index("griddepcontrol.wait") < idle.index("return;", idle.index("griddepcontrol"))


def test_the_acceptance_walk_waits_for_the_sweep_in_refused_sequences_too():
    walk = _body(_source("accept_compact.cu"), "accept_walk_kernel(")
    refused = _body(walk, "if (N < 1)")
    assert 0 < refused.index("griddepcontrol.wait") < refused.rindex("return;")


def test_who_may_take_it_ahead_of_the_wait():
    """The early mode (the caller's promise), and the call that has just launched its own work list."""
    launch = _body(_source(), "bool tree_attention_tc_launch(")
    assert re.findall(r"p\.tmem_first = ([^;]*);", launch) == ["p.early", "1"]
    assert re.search(r"attn_worklist_kernel<<<.*?p\.early = 0;\s*p\.tmem_first = 1;", launch, flags=re.S)


def test_kernel_attributes_are_remembered_per_context():
    """They hold for one device: a process that drives two has a context on each."""
    launch = _body(_source(), "bool tree_attention_tc_launch(")
    assert "cudaFuncSetAttribute" in launch and not re.search(r"\bstatic\b", launch)
