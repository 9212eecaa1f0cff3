"""CPU check of the rule that chained launches rest on: every kernel waits for the kernel before it ahead of its first access
to global memory and of its first return (the next kernel takes its completion for that of all earlier ones)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_01337_b200", "csrc")


def _closing(text, at, pair):
    """Index just past the bracket that closes the one at text[at]."""
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i + 1
    raise ValueError("unbalanced brackets")


def _kernels(source):
    """(name, parameters, body) of every __global__ function of a CUDA source."""
    source = re.sub(r"/\*.*?\*/", " ", source, flags=re.S)
    source = re.sub(r"//[^\n]*", " ", source)
    out = []
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^()]*\)\s*)?(\w+)\s*\(", source):
        end = _closing(source, m.end() - 1, "()")
        body = source.index("{", end)
        assert source[end:body].strip() == "", m.group(1)  # a definition, not a declaration
        out.append((m.group(1), source[m.end():end - 1], source[body + 1:_closing(source, body, "{}") - 1]))
    assert len(out) == len(re.findall(r"\b__global__\b", source))
    return out


def _fault(params, body):
    """What a kernel does ahead of its wait that it must not do, or None."""
    if re.match(r"\s*chain_begin\(\);", body):
        return None
    waits = [m.start() for m in re.finditer(r"\bchain_(?:wait|begin)\(\);", body)
             if body.count("{", 0, m.start()) == body.count("}", 0, m.start())]
    if not waits:
        return "never waits (outside a branch)"
    head = body[:waits[0]]
    found = re.search(r"\breturn\b|\batomic\w+|\btma_\w+|\bcp\.async|\b(?:ld|st|red)\.global", head)
    if found:
        return f"{found.group(0)} ahead of the wait"
    for p in re.split(r",", params):
        name = re.search(r"(\w+)\s*$", p)
        if name is None:
            continue
        use = rf"(?<![.\w]){name.group(1)}\b" if "*" in p else rf"\b{name.group(1)}\.[\w.]*\s*\[|\*\s*{name.group(1)}\b"
        if re.search(use, head):
            return f"uses {name.group(1)} ahead of the wait"
    return None


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_every_kernel_waits_before_it_touches_memory_or_returns(path):
    with open(path) as f:
        faults = {name: why for name, params, body in _kernels(f.read()) for why in [_fault(params, body)] if why}
    assert not faults


def test_the_begin_of_a_chained_kernel_waits():
    with open(os.path.join(CSRC, "c2r_common.cuh")) as f:
        text = f.read()
    assert re.search(r"void chain_begin\(\) \{[^}]*chain_wait\(\);", text)
    assert re.search(r"void chain_wait\(\) \{[^}]*griddepcontrol\.wait;", text)


@pytest.mark.parametrize("body,ok", [
    ("chain_begin(); x[0] = 1;", True),
    ("const int t = threadIdx.x; if (t == 0) { s = 0; } chain_wait(); x[t] = p.counts[t];", True),
    ("x[0] = 1;", False),
    ("if (n > 0) { chain_wait(); } x[0] = 1;", False),
    ("if (n > 0) return; chain_wait();", False),
    ("const int c = p.counts[0]; chain_wait(); x[0] = c;", False),
    ("x[0] = 1; chain_begin();", False),
])
def test_the_check_itself(body, ok):
    name, params, text = _kernels("__global__ void __launch_bounds__(64) k(int* __restrict__ x, int n, const P p) {" + body + "}")[0]
    assert name == "k" and (_fault(params, text) is None) == ok
