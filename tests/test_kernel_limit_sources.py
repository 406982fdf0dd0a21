"""Attribute calls cost about as much host time as a launch: what a training
evaluation sets of its kernels is set once per training set, not per evaluation."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_08119_gb300", "csrc")


def _block(s, start):
    """From the first brace at or after `start` to the one that closes it."""
    i = s.index("{", start)
    depth = 0
    for j in range(i, len(s)):
        depth += {"{": 1, "}": -1}.get(s[j], 0)
        if depth == 0:
            return s[i:j + 1]
    raise AssertionError("unbalanced braces")


def test_limits_are_set_once_per_training_set():
    with open(os.path.join(CSRC, "nep_train.cu")) as f:
        s = re.sub(r"//[^\n]*", "", f.read())
    body = _block(s, s.index("int prepare_evaluation("))
    once = _block(body, body.index("if (!ds->aux)"))
    setters = re.compile(r"cudaFuncSetAttribute|set_kernel_limits\(|prepare_owner_tc\(|prepare_pop_tc\(")
    assert setters.search(once)
    assert not setters.search(body.replace(once, ""))
    # nowhere else but in the function that this block calls
    assert not re.search(r"cudaFuncSetAttribute", s.replace(_block(s, s.index("int set_kernel_limits(")), ""))
