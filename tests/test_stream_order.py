"""Every handle works on a non-blocking stream, which the legacy stream's
copies and clears are not ordered with: what kernels of the handle read or
write must be set on the handle's stream.  Writes to device memory by the
legacy calls are therefore limited to the upload of X in sap_create (ordered
with the caller's own work) and the copies out to caller-owned buffers, each
followed by a wait."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1807_03425_gb300", "csrc")
ALLOWED = re.compile(r"^(h->X64|h->X32|tmp|dev \+|Yh_out|Yl_out)")


def test_no_legacy_stream_writes_beside_the_handles_stream():
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = open(os.path.join(CSRC, f)).read()
        assert not re.search(r"\bcudaMemset\(", src), f
        for m in re.finditer(r"\bcudaMemcpy\((([^;]|\n)*?)\);", src):
            if "DeviceToHost" in m.group(1) or "D2H" in m.group(1):
                continue
            assert ALLOWED.match(m.group(1).strip()), "%s: cudaMemcpy(%s" % (f, m.group(1))
