"""Kernels that fetch weights ahead of their wait for the kernel in front rely on that kernel having released them no earlier than its own
wait: only then is everything further ahead in the stream complete.  A cooperative kernel gains nothing from an earlier release (its CTAs
keep their SM to the end), so those that wait for a kernel in front before their first request release behind that wait."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_09323_b200", "csrc")


def _kernel(file, name):
    text = open(os.path.join(CSRC, file)).read()
    start = re.search(r"__global__ void [^{;]*\b%s\b" % name, text).start()
    end = text.find("\n}\n", start)
    return re.sub(r"//[^\n]*", "", text[start:end])


def test_the_cooperative_decode_kernel_waits_before_it_releases():
    body = _kernel("decode_coop.cuh", "decode_coop_kernel")
    assert body.count("pdl_wait()") == body.count("pdl_launch_dependents()") == 1
    assert body.index("pdl_wait()") < body.index("pdl_launch_dependents()")
    assert body.index("pdl_wait()") < body.index("request(p.wg")


def test_the_overlapped_selector_waits_before_it_releases():
    body = _kernel("small_batch.cuh", "sb_select_kernel")
    overlapped = body[body.index("if (BITS)"):body.index("} else {")]
    assert overlapped.index("pdl_wait()") < overlapped.index("pdl_launch_dependents()")
