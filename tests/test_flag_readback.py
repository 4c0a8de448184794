"""The tiles' error flags reach the host after every kernel that can set them (source level, CPU).

Kernels of both streams of an evaluation set the flags; the copy to the host is made on the caller's
stream, so it must be queued behind that stream's wait for the near field's."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_10059_gb300", "csrc",
                   "sph_api.cu")


def test_flags_are_copied_after_the_streams_join():
    s = re.sub(r"//[^\n]*", "", open(SRC).read())
    body = s[s.index("int fmm_queue(sph_ctx *c"):]
    body = body[:body.index("\n}\n")]
    join = body.index("cudaStreamWaitEvent(c->stream, c->near_join")
    copies = [m.start() for m in re.finditer(r"cudaMemcpyAsync\([^;]*S\.err[^;]*cudaMemcpyDeviceToHost", body)]
    mapped = body.index("fmm_near_add(")
    assert copies and all(p > join for p in copies)
    assert mapped > join
