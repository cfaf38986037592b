"""What the kernels of a chained step write (cell tables, accumulators, state, scale, moments) is not read through the
read-only path (__ldg, ld.global.nc), which takes its data to be constant while a kernel runs: a chained kernel can be
resident while the one that writes them still runs."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_11998_gb300", "csrc")
WRITTEN = ("cell64", "cdat", "cdB", "acc", "Bref", "scale", "a.I", "out.", "mscratch", "facc")


def call_arguments(text, name):
    """The argument text of every call of `name`."""
    for m in re.finditer(re.escape(name) + r"\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield m.start(), text[m.end():i - 1]


def origin(text, at, expr):
    """The initialiser of the pointer an argument starts with: the last `<name> = ...;` before it."""
    name = re.match(r"\s*&?\s*(\w+)", expr).group(1)
    inits = re.findall(r"\b%s\s*=\s*([^;]*);" % name, text[:at])
    return inits[-1] if inits else ""


@pytest.mark.parametrize("source", ["molc_fp64.cu", "molc_kernels.cu"])
def test_read_only_loads_take_plan_constants(source):
    text = open(os.path.join(CSRC, source)).read()
    calls = list(call_arguments(text, "__ldg"))
    assert calls
    for at, arg in calls:
        for w in WRITTEN:
            assert w not in arg and w not in origin(text, at, arg), (source, arg)
