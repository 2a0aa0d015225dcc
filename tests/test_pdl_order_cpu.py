"""Order of memory in the chains of line sweeps that follow one another by
programmatic launch (fv_mg.cu), from the source and without a GPU.

A kernel launched that way may start once every block of its predecessor has
triggered (or returned); only its wait makes the predecessor complete and its
stores visible.  What it reads ahead of the wait has to come from a kernel that
is complete by then: for sweeps that fetch b early, from the kernel that wrote
b.  The model below says which kernels are complete when one starts."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1704_08521_gb300", "csrc")


def _body(text, start):
    """The brace-balanced block that opens after `start`."""
    i = text.index("{", text.index(start))
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def _complete_at_start(kernels):
    """Per kernel of the list the set of earlier ones that are complete, and
    visible, when it starts.  A kernel is "plain", or programmatic and named by
    where it lets its successor in: "trigger-first" or "wait-first"."""
    done = []
    for i, k in enumerate(kernels):
        if k == "plain":                                   # starts when all that came before has ended
            done.append(set(range(i)))
        elif kernels[i - 1] == "trigger-first":            # no more than the predecessor itself started with
            done.append(set(done[i - 1]))
        else:                                              # its wait has returned (a plain one had none to make)
            done.append(set(range(i - 1)))
    return done


def test_model():
    # the first sweep starts beside the tail of the kernel before it, the second
    # one too if the first lets it in before waiting
    assert 0 not in _complete_at_start(["plain", "trigger-first", "trigger-first"])[2]
    assert 0 in _complete_at_start(["plain", "wait-first", "wait-first"])[2]
    assert _complete_at_start(["plain", "wait-first", "plain"])[2] == {0, 1}


def test_sweeps_fetch_b_from_a_complete_kernel():
    src = open(os.path.join(CSRC, "fv_mg.cu")).read()
    line = _body(src, "k_line(LevDev L")
    line = re.sub(r"//[^\n]*", "", line)
    wait, trigger = line.index("pdl_wait()"), line.index("pdl_trigger()")
    assert line.count("pdl_wait()") == line.count("pdl_trigger()") == 1
    sweep = "trigger-first" if trigger < wait else "wait-first"
    # b is read ahead of the wait only under b_early, x never
    head = line[:wait]
    assert re.search(r"if \(b_early\)[^;]*= b\[c\];", head) and len(re.findall(r"\bb\[", head)) == 1
    assert not re.search(r"\bx\[", head)
    # the V-cycle clears b_early for the sweep after the kernel that wrote b
    cycle = _body(src, "fv_status vcycle(")
    assert "bool b_early = false;" in cycle and cycle.count("b_early = true;") == 1
    chain = ["plain"] + 6 * [sweep]                        # restriction (b), then x, y, z in two colours
    early = [False, False] + 5 * [True]
    for i, done in enumerate(_complete_at_start(chain)):
        assert not early[i] or 0 in done, f"sweep {i} reads b while the kernel that writes it may be running"
