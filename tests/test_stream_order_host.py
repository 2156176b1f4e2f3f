"""Device memory is written on the bound stream: a cudaMemcpy from pageable host memory may return
before its transfer has ended, and work on a non-blocking stream does not wait for it."""
import glob
import os
import re

import paper_2605_30583_gb300

CSRC = os.path.join(os.path.dirname(paper_2605_30583_gb300.__file__), "csrc")


def test_no_upload_outside_the_stream():
    found = []
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = open(f).read()
        found += [(os.path.basename(f), m.group(0)) for m in re.finditer(r"\bcudaMemcpy\s*\([^;]*?;", text)
                  if "HostToDevice" in m.group(0)]
    assert not found
