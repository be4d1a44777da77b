"""Host-side copies into device arrays are ordered on the handle's stream.

Handles run on non-blocking streams, which do not wait for the legacy default stream: a plain cudaMemcpy of
a pageable buffer may return once the buffer is staged and a plain cudaMemset returns at once, so a kernel
launched on the handle's stream after either may read the array before the data arrive.  A lost race shows as
wrong constants kept for the life of the handle, not as an error, so the order is checked in the source."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_13190_gb300", "csrc")


def source(name):
    src = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", src, flags=re.S))


def calls(src, name):
    """The argument texts of every call of `name`."""
    out = []
    for m in re.finditer(r"\b%s\(" % name, src):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(src[i], 0)
            i += 1
        out.append(" ".join(src[m.end():i - 1].split()))
    return out


def test_copies_to_the_device_are_ordered_on_the_handles_stream():
    src = source("ldpm_api.cu")
    # the law hook has no handle: its copies and its kernel are all on the legacy default stream
    handle, hook = src.split("int ldpm_facet_law_vjp(")
    assert re.search(r"launch_law_vjp<double>\([^;]*, 0\);", hook)
    late = [c for c in calls(handle, "cudaMemcpy") if "cudaMemcpyDeviceToHost" not in c]
    assert not late, late
    assert not calls(handle, "cudaMemset"), calls(handle, "cudaMemset")
    n = 0
    for name in ("cudaMemcpyAsync", "cudaMemsetAsync", "cudaMemcpy2DAsync"):
        for c in calls(handle, name):
            assert c.endswith("h->stream"), (name, c)
            n += 1
    assert n > 10
