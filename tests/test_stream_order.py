"""Every copy, fill and kernel launch of the library names its stream.  The
library's streams are non-blocking: work on the default stream is not ordered
with theirs, and a blocking copy from pageable memory returns once its source is
staged, not when the data has arrived on the device."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _code():
    for f in sorted(glob.glob(os.path.join(ROOT, "paper_1401_0782_gb300", "csrc", "*.cu*"))):
        txt = re.sub(r"/\*.*?\*/", "", open(f).read(), flags=re.S)
        yield os.path.basename(f), re.sub(r"//[^\n]*", "", txt)


def test_copies_and_fills_name_a_stream():
    bad = [(f, m.group(0)) for f, txt in _code() for m in re.finditer(r"\bcuda(Memcpy|Memset)(2D|3D|ToSymbol)?\s*\(", txt)]
    assert not bad, bad


def test_launches_name_a_stream():
    n = 0
    for f, txt in _code():
        for m in re.finditer(r"<<<(.*?)>>>", txt, flags=re.S):
            n += 1
            assert re.search(r",\s*(c->)?st\w*\s*$", m.group(1)), (f, m.group(0))
    assert n > 20
