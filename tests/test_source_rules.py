"""Rules of the CUDA sources that a reader can check and a run cannot: a run
passes whenever the compiler happens to keep a warp together."""
import glob
import os
import re

from paper_2605_28283_gb300 import build


def test_aligned_instructions_follow_a_syncwarp():
    """`.aligned` instructions (tcgen05 allocation and TMEM loads, named
    barriers) are undefined for a warp whose lanes have come apart.  Each stands
    in a helper of its own that brings the lanes together first."""
    found = 0
    for path in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r'"[^"\n]*(\.sync\.aligned|\bbar\.(sync|red|arrive))', text):
            start = text.rfind("PP_DEVINL", 0, m.start())
            body = text[text.index("{", start):m.start()]
            assert start >= 0 and re.match(r"\{\s*__syncwarp\(\);\s*(unsigned r;\s*)?asm volatile\(", body), \
                (os.path.basename(path), text[start:m.start() + 60])
            found += 1
    assert found >= 9


def test_union_kernel_reads_nothing_before_the_previous_kernel_is_done():
    """Launched with programmatic dependent launch, the union kernel may run while
    the previous kernel on the stream writes any of its inputs, W_r among them: up
    to pdl_wait() it only prefetches into L2."""
    text = open(os.path.join(build.CSRC, "union.cu")).read()
    router = re.sub(r"//[^\n]*", "", text[text.index("PP_DEVINL void router_phase("):text.index("PP_DEVINL void select_phase(")])
    before = router[:router.index("pdl_wait()")]
    assert "tma_prefetch_2d(&a.map_wr" in before
    assert not re.search(r"tma_load_2d|bulk_g2s|ld_relaxed|__ldg|__ldcg|\ba\.part\b", before)
