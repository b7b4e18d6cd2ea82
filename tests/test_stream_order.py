"""Order of host-to-device copies, read from the source.  The library's streams are non-blocking: work on them does
not wait for the default stream, and a plain cudaMemcpy of pageable memory may return while its copy to the device is
still under way.  So tables that a kernel reads are copied on the stream that launches it (cudaMemcpyAsync), never
with the default-stream copy."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_07929_gb300", "csrc")


def test_no_upload_on_the_default_stream():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\bcudaMemcpy(?:2D|3D)?\s*\(([^;]*?);", text, flags=re.S):
            if "HostToDevice" in m.group(1) or "cudaMemcpyDefault" in m.group(1):
                found.append((os.path.basename(path), m.group(0)))
    assert not found, found
