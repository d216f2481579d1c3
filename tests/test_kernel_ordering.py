"""Orderings that a kernel has to ask for and that no result shows reliably, read off the sources:
an accumulator in tensor memory is handed from its readers to the next MMA between two tcgen05
fences, and a kernel that may start early makes no invariant loads."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_10514_gb300", "csrc")


def code(name):
    """A source file without its comments."""
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", text), flags=re.S)


def function(text, head):
    """The body of the function that starts with `head`."""
    at = text.index("{", text.index(head))
    depth, i = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at:i + 1]
        i += 1


def test_issuer_fences_after_every_wait():
    text = code("gemm_oz.cu")
    issuer = text[text.index("elect_lane()"):]
    issuer = issuer[:issuer.index("setmaxnreg.inc")]
    waits = [m.start() for m in re.finditer(r"bar_poll\w*\(", issuer)]
    assert len(waits) == 2  # a stage, an accumulator
    for w in waits:
        rest = issuer[w:]
        assert rest.index("tcgen05.fence::after_thread_sync") < rest.index("mma_pair("), rest[:60]


def test_accumulator_is_handed_over_between_fences():
    """Readers: wait::ld, fence::before_thread_sync, arrival at cluster scope; issuer: a wait at
    cluster scope (and the fence of the test above)."""
    oz, helpers = code("gemm_oz.cu"), code("tcgen05.cuh")
    drain = function(oz, "auto drain = [&]")
    order = [drain.index(x) for x in ("tcgen05.wait::ld", "tcgen05.fence::before_thread_sync", "__syncwarp()",
                                      "arrive_remote(")]
    assert order == sorted(order)
    assert re.search(r"mbarrier\.arrive\.\w+\.cluster\.shared::cluster", function(helpers, "void arrive_remote("))
    assert "acquire.cluster" in function(helpers, "bool bar_test_cluster(")
    assert re.search(r"bar_poll_cluster\(&cfree\[", oz)


def test_dependent_kernels_make_no_invariant_loads():
    """A kernel that may be placed before the launch before it has ended (it calls dep_wait) reads
    what that launch writes: an invariant load (__ldg, or through const __restrict__, also of a
    function that it calls) may be moved above the wait."""
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        text = code(name)
        if name == "common.cuh" or "dep_wait(" not in text:
            continue
        seen += 1
        assert "__ldg(" not in text, name
        assert not re.search(r"const\s+\w+(<\w+>)?\s*\*\s*__restrict__", text), name
    assert seen >= 6
