"""sm_state_create frees what it allocated when a later step of it fails.

The failing calls cannot be provoked without a device, so this reads the
source: the function that owns the new state has one way out per outcome, and
what can fail runs in a function of its own that returns a status."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_04998_gb300", "csrc")


def body(src, head):
    """Text of the function that starts with `head`, comments removed."""
    i = src.index("{", src.index(head))
    depth = 0
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth == 0:
            return re.sub(r"//[^\n]*", "", src[i:j + 1])


def test_no_early_return_between_the_state_and_its_release():
    with open(os.path.join(CSRC, "integrate.cu")) as fh:
        create = body(fh.read(), "sm_status sm_state_create(const sm_net* net")
    after = create[create.index("new (std::nothrow) sm_state()"):]
    # (the macro returns from the function that it stands in)
    assert "SM_TRY_CUDA" not in after
    returns = re.findall(r"return ([^;]+);", after)
    assert returns == ["SM_ENOMEM", "r", "SM_OK"], returns
    assert re.search(r"free_state\(st\);\s*delete st;\s*return r;", after)
    # set-up on the state's own stream: kernels on it do not wait for the legacy one
    assert "cudaMemset(" not in create


def test_state_is_cleared_on_its_own_stream():
    with open(os.path.join(CSRC, "integrate.cu")) as fh:
        src = re.sub(r"//[^\n]*", "", fh.read())
    assert not re.search(r"\bcudaMemset\(", src)
