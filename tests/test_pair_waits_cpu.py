"""A pair's barriers collect arrivals of both of its CTAs, and a wait whose scope is one CTA does not order what the partner did before
it arrived.  Read from the source: every wait of the prefill kernel is at cluster scope for a pair, except on the barriers of the
packed ring, whose arrivals are the CTA's own."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_24011_b200", "csrc")


def test_scope_of_the_waits():
    s = open(os.path.join(CSRC, "aq_gemm.cu")).read()
    kernel = s[s.index("__device__ __forceinline__ bool dequant_slab("):s.index("tensor_map_encoder() {")]
    waits = re.findall(r"mbar_wait(?:_warp)?<([^>]*)>\((bar_[a-z]+)", kernel)
    assert sorted(b for _, b in waits) == sorted("bar_" + n for n in ("aempty", "pfull", "dfull", "bempty", "pempty", "dempty", "afull", "bfull"))
    for args, bar in waits:
        assert args == ("PAIR, true" if bar in ("bar_pfull", "bar_pempty") else "PAIR"), (bar, args)
    assert "template <bool PAIR, bool OWN = !PAIR>\n__device__ __forceinline__ bool mbar_wait(" in s
    assert "OWN ? mbar_try(bar, parity) : mbar_try_cluster(bar, parity)" in s
    wrapper = open(os.path.join(CSRC, "aq_tc.cuh")).read()
    body = wrapper[wrapper.index("bool mbar_try_cluster("):]
    assert "mbarrier.try_wait.parity.acquire.cluster." in body[:body.index("}\n")]
