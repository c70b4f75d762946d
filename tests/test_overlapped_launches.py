"""Kernels that are set up while the kernel before them still runs read nothing through the read-only path: such loads ask
for data that is not written while the kernel is there, and may be moved above its wait."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_16673_b200", "csrc")


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", text), flags=re.S)


OVERLAPPED = [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cu")
              and re.search(r"\b(after_previous_kernel|wait_for_previous_kernel)\(\)", code(f))]


def test_which_files_have_overlapped_kernels():
    launched = [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cu") and re.search(r"\blaunch\(\w", code(f))]
    assert OVERLAPPED == launched and len(OVERLAPPED) >= 5


@pytest.mark.parametrize("name", OVERLAPPED)
def test_no_loads_through_the_read_only_path(name):
    text = code(name)
    assert not re.findall(r"__ldg|ld\.global(?:\.\w+)*\.nc|const\s+[\w:]+\s*\*\s*__restrict__", text)


@pytest.mark.parametrize("name", OVERLAPPED)
def test_every_overlapped_kernel_waits_first(name):
    """The wait stands before any access to global memory: at the top of the body, but for the form of the effective-query
    kernel that sets up its barriers and asks for tiles beforehand."""
    text = code(name)
    for kernel in set(re.findall(r"\blaunch\((\w+_kernel)", text)):
        body = text[re.search(r"\b%s\(" % kernel, text).end():]
        body = body[body.index("{") + 1:]
        if kernel == "verify_effective_kernel":
            assert body.index("wait_for_previous_kernel()") < body.index("p.ws.") and \
                body.index("wait_for_previous_kernel()") < body.index("p.node_offsets")
        else:
            assert body.lstrip().startswith("after_previous_kernel();"), kernel
