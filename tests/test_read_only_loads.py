"""Where the kernels use the read-only load path.  Its contract is that nobody
writes the memory while the kernel runs.  A chained kernel may start while its
predecessor still writes, so there it may only touch what the caller handed in."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_09703_gb300", "csrc")
# file -> what read-only loads may read: targets and the forward's row statistics
# (arguments of a call, complete before its first kernel starts)
INPUTS = {"mls_head.cu": (r"p\.y\b", r"p\.stats\b"), "mls_reduce.cu": (r"y$",)}


def read_only_operands(text):
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__ldg\s*\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text[m.end():i - 1]
    for m in re.finditer(r"__restrict__\s+(\w+)", text):
        yield m.group(1)
    for m in re.finditer(r"ld\.global\S*\.nc\S*", text):
        yield m.group(0)


def test_chained_kernels_read_only_the_callers_inputs_that_way():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(path).read()
        name = os.path.basename(path)
        if "launch_chained(" not in text:
            continue
        for operand in read_only_operands(text):
            seen += 1
            assert any(re.match(r"\W*(?:reinterpret_cast<[^>]*>\()?" + ok, operand)
                       for ok in INPUTS.get(name, ())), f"{name}: {operand}"
    assert seen >= 4


def test_junction_loads_allow_gradients_over_inputs():
    """d_o may be o and d_e may be e, so nothing the junction reads stays unwritten."""
    with open(os.path.join(CSRC, "mls_junction.cu")) as f:
        assert list(read_only_operands(f.read())) == []
