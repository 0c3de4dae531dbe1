"""Host tables and fills go through the stream whose kernels read them: a plain cudaMemcpy or cudaMemset
runs on the legacy stream, which a stream created non-blocking does not wait for."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1410_3584_gb300", "csrc")


def test_no_upload_or_fill_on_the_legacy_stream():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        with open(path, encoding="utf-8") as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"\bcudaMemset\s*\(|\bcudaMemcpy\s*\([^;]*?cudaMemcpy(HostToDevice|DeviceToDevice|Default)", text):
            found.append("%s: %s" % (os.path.basename(path), m.group(0)[:60]))
    assert not found, found
