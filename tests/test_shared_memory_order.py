"""Shared memory that one thread writes and another reads, in the source: stores into another CTA's shared memory come after all
CTAs of the cluster have started, and are waited for before they are read; between the lanes of a warp stands a __syncwarp, since
votes and reductions order no memory."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_16673_b200", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", text), flags=re.S)


def block(text, start):
    """What stands between the first brace after `start` and its match."""
    begin = text.index("{", start) + 1
    depth, i = 1, begin
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[begin:i - 1]


def function(name, func):
    text = code(name)
    return block(text, re.search(r"\b%s\([^;{]*\)\s*\{" % func, text).start())


CLUSTERED = [(f, k) for f in SOURCES for k in re.findall(r"__cluster_dims__\([^)]*\)\s*__launch_bounds__\([^{;]*?\)\s*(\w+)\(", code(f))]


def test_which_kernels_use_other_ctas_memory():
    assert CLUSTERED and sum(code(f).count("mapa.") for f in SOURCES) == sum(function(*c).count("mapa.") for c in CLUSTERED)


@pytest.mark.parametrize("name,kernel", CLUSTERED)
def test_other_ctas_have_started_before_their_memory_is_written(name, kernel):
    """Every thread arrives and waits before the first remote address is formed, and once more behind the last remote store."""
    text = function(name, kernel)
    first, last = text.index("mapa."), text.rindex("st.shared::cluster")
    for part in (text[:first], text[last:]):
        arrive, wait = part.index("barrier.cluster.arrive"), part.index("barrier.cluster.wait")
        assert arrive < wait
    assert not re.search(r"\breturn;", text[:last])                 # nobody leaves before
    assert "release" in text[last:].split("barrier.cluster.arrive")[1][:20]
    assert "acquire" in text[last:].split("barrier.cluster.wait")[1][:20]


# file, function, how the loop around both starts (None: they follow one another), the write, the read by other lanes
HANDED_OVER = [
    ("plan.cu", "accept_kernel", None, "target[t] = target_tok[base + t];", "target[p];"),
    ("plan.cu", "accept_kernel", None, "step[t] = ", "a = step[a];"),
    ("plan.cu", "stochastic_accept_kernel", None, "first[t] = kStochNodes;", "atomicMin(&first"),
    ("plan.cu", "stochastic_accept_kernel", None, "atomicMin(&first", "first[pa + 1] != a"),
    ("plan.cu", "prune_small_kernel", None, "q[lane + 32 * k] = mine[k];", "q[par[k]]"),
    ("plan.cu", "prune_small_kernel", "while (done", "q[lane + 32 * k] = mine[k];", "q[par[k]]"),
    ("plan.cu", "prune_small_kernel", "while (done", "q[par[k]]", "q[lane + 32 * k] = mine[k];"),
    ("effective.cu", "plan_paths", None, "par[i] = int8_t(pa);", "write_path("),
    ("effective.cu", "plan_paths", "for (int b = warp;", "write_path(", "par[i] = int8_t(pa);"),
]


@pytest.mark.parametrize("name,func,loop,write,read", HANDED_OVER)
def test_lanes_synchronise_between_writing_and_reading(name, func, loop, write, read):
    text = function(name, func)
    if loop:
        text = 2 * block(text, text.index(loop))                     # one turn and the next
        text = text[text.index(write):]
    between = text[text.index(write):]
    between = between[:between.index(read)]
    assert re.search(r"__sync(warp|threads)\(\)", between)
