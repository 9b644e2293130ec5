"""What cannot be provoked on a GPU without risking a fault or a hang, held in the
kernels' sources (no GPU): the memory order of hand-overs between SMs, and that a
warp which gives up a wait does so as a whole."""
import os
import re

import pytest

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


@pytest.mark.parametrize("name", ["herk_tc.cu", "zherk_tc.cu", "mlp_tc.cu", "mlp_train_tc.cu", "mlp_chain_tc.cu",
                                  "mlp_wgrad_tc.cu"])
def test_warps_that_read_tensor_memory_give_up_together(name):
    # tcgen05.ld needs the whole warp: a wait that ran out in one lane only, or an
    # abort flag that one lane alone has seen, must not part the warp in front of it
    s = source(name)
    reads = [m.start() for m in re.finditer(r"\b(?:tmem_ld\d+|drain_layer)\(", s)]
    waits = [(m.start(), m.group(1)) for m in re.finditer(r"\b(wait_\w+)\((?!uint32_t|auto)", s)]
    waits = [w for w in waits if w[1].startswith(("wait_bounded", "wait_warp"))]
    checked = 0
    for r in reads:
        before = [w for at, w in waits if at < r]
        if not before:  # (a helper, defined above the kernel that waits)
            continue
        assert before[-1].startswith("wait_warp"), s[r - 200:r]
        checked += 1
    assert checked
    assert not re.search(r"\*abort_flag\) (?:break|\{ ok = false)", s)


def test_warp_waits_vote():
    s = source("tc.cuh")
    for name in ("wait_warp", "wait_warp_spin"):
        body = s[s.index(f"bool {name}("):]
        body = body[:body.index("}")]
        assert re.search(r"return __all_sync\(0xffffffffu, wait_bounded\w*\(", body), name
    assert re.search(r"bool warp_aborted\([^)]*\) \{ return __any_sync\(0xffffffffu, \*abort_flag != 0\)", s)


def _poly(text, name):
    """The FP32 literals of the statement that sets `name`, in order."""
    i = text.index(name)
    return [float(v) for v in re.findall(r"(-?\d+\.\d+)f", text[i:text.index(";", i)])]


def test_packed_sincos_has_the_pinned_coefficients():
    # the streamed schedule's packed cos / sin holds the polynomials of zcore.cuh,
    # whose error bound tests/test_oracle_pins.py checks
    z, p = source("zcore.cuh"), source("zherk_tc.cu")
    z, p = z[z.index("cos_sin_turns"):], p[p.index("cos_sin_turns2("):]
    sin, cos = _poly(z, "const float sp"), _poly(z, "const float cp")
    assert len(sin) == 4 and len(cos) == 5
    assert _poly(p, "const F2 sp") == sin
    assert _poly(p, "const F2 cp") == cos


def test_no_kernel_launch_assumes_a_number_of_sms():
    for name in sorted(os.listdir(CSRC)):
        assert not re.search(r"\b152\b", source(name)), name
