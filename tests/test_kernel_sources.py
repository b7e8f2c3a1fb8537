"""Rules that the kernels keep and that no run without a fault can show: checked in their source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_05858_b200", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_bounded_waits_are_answered_by_the_warp():
    """Every role of the tensor-core kernel runs warp-wide instructions behind its waits, so a wait that runs out, or a failure of
    another role, has to part no lanes: each wait's result goes through a vote, and the failure flag is read through one or once all
    roles have met."""
    text = source("bconv_tc.cu")
    warp_wait = text[text.index("bool mbar_wait_warp("):]
    warp_wait = warp_wait[:warp_wait.index("\n}")]
    assert "if (__all_sync(0xFFFFFFFFu, done != 0)) return true;" in warp_wait and "__any_sync(0xFFFFFFFFu, *fail != 0)" in warp_wait
    kernel = text[text.index("bconv_tc_kernel("):text.index("tc_prepare_weights_kernel")]
    # the role that issues the MMAs: a whole warp, or one lane of a pair's leader
    assert "if (rank == 0 && (!PAIR || lane == 0)) {" in kernel
    assert "return PAIR ? mbar_wait_lane_cluster(bar, parity, s_fail, g.wait_polls) : mbar_wait_warp(bar, parity, s_fail, g.wait_polls);" in kernel
    kernel = kernel.replace("PAIR ? mbar_wait_lane_cluster(", "").replace("mbar_wait_warp(", "").replace("PAIR ? *s_fail != 0 : ", "")
    calls = [m.start() for m in re.finditer(r"\bmbar_wait\w*\(", kernel)]
    assert len(calls) >= 5
    for at in calls:
        vote = kernel.rfind("__all_sync(0xFFFFFFFFu", 0, at)
        assert vote >= 0 and ";" not in kernel[vote:at], kernel[max(0, at - 200):at + 100]
    for m in re.finditer(r"\*s_fail != 0", kernel):
        line = kernel[kernel.rfind("\n", 0, m.start()) + 1:kernel.index("\n", m.end())]
        assert "__any_sync(0xFFFFFFFFu, *s_fail != 0)" in line or "*s_fail != 0 && tid == 0" in line, line


def test_pointers_to_the_previous_kernel_s_output_come_through_the_wait():
    """Loads through a const __restrict__ pointer count as invariant and may move above a chained launch's wait.  In the packs, whose
    input is such a pointer, the wait therefore hands out the pointer that is read."""
    text = source("pack.cu")
    kernels = [k for k in re.split(r"(?=template <|__global__)", text) if k.startswith("__global__") and "chain_trigger()" in k]
    assert len(kernels) == 6
    for k in kernels:
        assert "const T* __restrict__ x" in k and "x = chain_wait_for(x);" in k and "chain_wait();" not in k, k[:200]
        body = k[k.index("{"):]
        before = body[:body.index("x = chain_wait_for(x);")]
        assert not re.search(r"\bx\b", before), before


def test_packs_let_their_successor_in_behind_their_loads():
    """CTAs of the next kernel that come in while a pack's are still loading settle unevenly on the SMs (a third more time for a small
    convolution and its pack): in every pack the trigger stands behind the last read of the input, but for packs of few CTAs."""
    text = source("pack.cu")
    for k in [k for k in re.split(r"(?=template <|__global__)", text) if k.startswith("__global__") and "chain_trigger()" in k]:
        body = k[k.index("{"):]
        assert "if (room == 2) chain_trigger();\n  x = chain_wait_for(x);" in body
        if "pack_nhwc_c64" in k:  # (lets the next kernel in at its end)
            assert body.count("chain_trigger()") == 1
            continue
        assert body.count("chain_trigger()") == 2
        at = body.index("if (room == 1) chain_trigger()")
        assert not re.search(r"\b(x|xn|src|row)\s*(\[|\+)|ld_stream_v4\(|__ldcs\(", body[at:]), body[at:at + 200]
    assert "return 10 * ctas <= 3 * sms ? 2 : 1;" in text


def test_a_tensor_core_cta_has_its_sm_alone():
    """Every launch asks for more shared memory than two CTAs of an SM can have: each takes all of the tensor memory there."""
    text = source("bconv_tc.cu")
    assert "static_assert(2 * (TC_SMEM_ALONE + 1024) > 228 * 1024" in text
    launch = text[text.index("dabnn_status tc_launch(const TcArgs& g"):]
    assert launch.index("smem = TC_SMEM_ALONE;") < launch.index("<<<")
