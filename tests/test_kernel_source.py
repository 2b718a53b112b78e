"""Properties of the kernels that no run shows reliably, read from their source."""
import os
import re

import pytest

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


@pytest.mark.parametrize("kernel", ["tc_kernel(", "tc_pair_kernel("])
def test_exit_waits_for_the_last_mma_ignore_the_abort_flag(kernel):
    """The wait for the last commit stands between the MMAs and the release of shared and tensor memory (in a pair of
    CTAs also the other CTA's): after an abort it must not return early, as the waits of the roles do."""
    k = body(source("laph_tc.cu"), kernel)
    waits = re.findall(r"(\w+)\([^;]*&S->done, 0u\)", k)
    assert waits and set(waits) == {"drain_wait"}
    assert k.rindex("&S->done, 0u") < k.rindex("dealloc")
    if "pair" in kernel:   # CTA 0 waits before the CTAs meet, CTA 1 for the commit's arrival after that
        assert len(waits) == 2
        first, last = [m.start() for m in re.finditer(r"&S->done, 0u", k)]
        assert first < k.rindex("cluster_sync_all()") < last


def test_arrivals_between_the_ctas_of_a_pair_name_the_cluster_scope():
    """Without a scope an mbarrier operation's is the CTA, which does not order it with the other CTA's.  CTA 1's half of B
    is written by its own copies, whose completion has to be counted in CTA 0: the MMA that CTA 0 issues reads it."""
    src = source("laph_tc.cu")
    arrives = re.findall(r"mbarrier\.arrive[\w.:]*shared::cluster\.b64", src)
    assert arrives and all(".release.cluster." in a or ".relaxed.cluster." in a for a in arrives)
    k = body(src, "tc_pair_kernel(")
    assert re.search(r"if \(rank\)\s*tma_b1\([^;]*peer_addr\(fb, 0\)\)", k)
    # barriers that the other CTA's threads or MMAs arrive on are waited for at cluster scope
    for bar in ("a_full", "acc_empty", "acc_full", "empty", "tempty"):
        assert not re.search(r"warp_wait\(c, &S->%s\[" % bar, k), bar
