"""Every copy and fill of the library is queued on the stream of its handle: the calls
without a stream order nothing against a non-blocking one, and from pageable
memory they may return before the data is on the device."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_copy_without_a_stream():
    found = []
    for path in glob.glob(os.path.join(ROOT, "paper_1003_3779_gb300", "csrc", "*")):
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        found += [(os.path.basename(path), m) for m in re.findall(r"\bcuda(?:Memcpy|Memset)\w*(?<!Async)\s*\(", src)]
    assert not found
