"""Order of the operator passes' dependency wait, read from their source: no
block of a pass leaves before the wait for the kernel it was launched behind,
so that a pass never completes before the passes ahead of it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1803_06237_gb300", "csrc")


def _body(text, at):
    """The braces' content of the first block that opens after `at`."""
    start = text.index("{", at)
    depth, i = 0, start
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start:i]
        i += 1


def _read(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("name,kernels", [("matvec.cu", 11), ("any_x.cuh", 2), ("any_b.cuh", 1)])
def test_no_pass_leaves_before_its_wait(name, kernels):
    text = _read(name)
    seen = 0
    for m in re.finditer(r"__global__ void[^;{]*?(\w+_kernel)\(([^{;]*?)\)\s*\{", text):
        if "PassPtrs" not in m.group(2):
            continue
        body = _body(text, m.end() - 1)
        wait = re.search(r"\b(skip_after_wait\(pp\)|pdl_wait\(\))", body)
        leave = re.search(r"\breturn\b\s*;", body)
        assert wait and (leave is None or wait.start() < leave.start()), m.group(1)
        seen += 1
    assert seen == kernels


def test_the_flag_is_read_behind_the_wait():
    text = _read("passes.cuh")
    body = _body(text, text.index("bool skip_after_wait"))
    assert body.index("pdl_wait()") < body.index("*(const volatile int*)f")
    assert body.count("*f") == 0 and body.count("*(") == 1 and body.count("pp.live") == 1   # its only read
    for name in ("matvec.cu", "any_x.cuh", "any_b.cuh"):
        assert not re.search(r"pp\.live(?!\[k\] = )", _read(name)), name
