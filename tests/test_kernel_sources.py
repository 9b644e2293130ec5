"""What cannot be provoked on a GPU without risking a fault or a hang, held in the
kernels' sources (no GPU): the memory order of hand-overs between SMs."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_09763_gb300", "csrc")


def source(name):
    """The source with its comments taken out and runs of blanks made one."""
    s = open(os.path.join(CSRC, name)).read()
    s = re.sub(r"//[^\n]*", "", s)
    return re.sub(r"\s+", " ", s)


def test_ring_counts_are_released_and_acquired():
    # a chunk of the ring is handed from the SMs that wrote it to those that load it
    # (ready), and back (done, then freed within an SM): a relaxed access on either
    # side leaves the stores and the loads unordered
    s = source("zherk_tc.cu")
    assert "ld.acquire.gpu" in s and "fence.acq_rel.gpu" in s
    kernel = s[s.index("k_zherk(const __grid_constant__"):s.index("k_zherk_prep(")]
    # the lanes that saw a count acquire it, and meet before one of them goes on
    assert re.search(r"if \(q \+ lane < have\) ld_acquire\(P\.ready \+ base \+ q \+ lane\); __syncwarp\(\); "
                     r"asm volatile\(\"fence\.proxy\.async\.global", kernel)
    assert re.search(r"if \(lane < adv\) ld_acquire\(P\.done \+ c\); __syncwarp\(\); "
                     r"if \(lane == 0\) st_release_cta\(freed, next\)", kernel)
    # every count an SM adds follows a fence, but for chunks that it never loads
    adds = [m.start() for m in re.finditer(r"red_add\(", kernel)]
    skipped = kernel.index("for (int q = len; q < wlen; ++q) red_add(P.done")
    fenced = kernel.index("fence_release(); if (built) red_add(P.ready + base + q, 1); "
                          "for (int i = 0; i < land; ++i) red_add(P.done")
    assert len(adds) == 3 and sum(skipped < a < skipped + 60 for a in adds) == 1
    assert sum(fenced < a < fenced + 150 for a in adds) == 2
    # the words in shared memory: their address, a release, an acquire each
    for word in ("freed", "landed"):
        assert len(re.findall(r"\b%s\b" % word, kernel)) == 3, word
        assert f"st_release_cta({word}" in kernel and f"ld_acquire_cta({word})" in kernel
    assert len(re.findall(r"P\.(?:ready|done)\b", kernel)) == 7
