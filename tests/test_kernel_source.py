"""Properties of the kernels that no run shows reliably, read from their source."""
import os
import re

from helpers import ROOT

CSRC = os.path.join(ROOT, "paper_2510_26313_gb300", "csrc")


def source(name: str) -> str:
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def body(src: str, head: str) -> str:
    """The parameter list and body of the function whose declaration ends in `head`."""
    a = src.index(head)
    depth, i = 0, src.index("{", a)
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth == 0:
            return src[a:j + 1]
    raise AssertionError(head)


def test_filter_vectors_are_not_promised_read_only():
    """A filter step is resident while the step before it writes its input vector: a const __restrict__ parameter or a
    read-only load would let the compiler move the loads above griddepcontrol.wait or make them non-coherent."""
    src = source("laph_lanczos.cu")
    k = body(src, "lap_soa_kernel(")
    params = k[:k.index("{")]
    assert re.findall(r"__restrict__\s*(\w+)", params) == ["Us"]
    assert "__restrict__" not in body(src, "load_site(").split("{")[0]
    assert "__ldg" not in body(src, "load_site(")
    # the first access to a vector comes after the wait
    assert k.index("griddepcontrol.wait") < k.index("load_site<")
