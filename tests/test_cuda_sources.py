"""Memory rules of the CUDA sources that no run can show to be broken: the
kernels of a dependent chain of launches may be running while the kernel
before them still writes."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_06161_gb300", "csrc")
CHAIN = ["binning.cu", "gauss.cu", "composite.cu", "deform_mlp.cu", "decoder.cu"]

# What the chains read through the non-coherent path: the caller's parameters,
# planes, weights and upstream gradients, none of them written by a pass
# (corners() and load_sh() read through p, the MLP's weight loads and the
# feature gradient through src).
INPUTS = {"p", "p + C / 4", "p + row", "p + row + C / 4", "p + i", "src + i", "src + d4",
          "reinterpret_cast<const float4*>(a.quats) + g", "a.wh + k * kHidden + o", "a.w2 + o * kHidden + o1",
          "a.w1 + o1 * C + c"} | {"a.means + 3 * (size_t)g" + s for s in ("", " + 1", " + 2")}


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _argument(text, start):
    depth, i = 1, start
    while depth:
        depth += {"(": 1, ")": -1}.get(text[i], 0)
        i += 1
    return " ".join(text[start:i - 1].split())


@pytest.mark.parametrize("name", CHAIN)
def test_chain_kernels_promise_no_constant_memory(name):
    text = _source(name)
    kernels = list(re.finditer(r"__global__\s", text))
    assert kernels
    waits = 0
    for m, end in zip(kernels, [k.start() for k in kernels[1:]] + [len(text)]):
        body = text.index("{", m.end())
        if "grid_dep_wait();" in text[body:end]:
            waits += 1
            assert "__restrict__" not in text[m.end():body], text[m.end():body]
    assert waits


@pytest.mark.parametrize("name", CHAIN)
def test_non_coherent_loads_read_inputs_only(name):
    text = _source(name)
    for m in re.finditer(r"__ldg\(", text):
        assert _argument(text, m.end()) in INPUTS, _argument(text, m.end())


def test_inline_memory_accesses_are_ordered():
    # An instruction with an address operand is tied to the stores before it
    # only by the clobber (a prefetch moves no data).
    accesses = 0
    for name in sorted(os.listdir(CSRC)):
        text = _source(name)
        for m in re.finditer(r"\basm(?:\s+volatile)?\s*\(", text):
            stmt = _argument(text, m.end())
            if re.search(r"\[%", stmt) and not stmt.startswith('"prefetch'):
                accesses += 1
                assert '"memory"' in stmt, (name, stmt)
    assert accesses > 20
