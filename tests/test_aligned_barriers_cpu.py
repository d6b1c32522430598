"""Barriers and TMEM loads in their .aligned forms must be executed by a warp's
threads together; after a branch that depends on the lane nothing but an
explicit __syncwarp() promises that.  No run can show the lack of one (the
compiler mostly reconverges by itself), so the sources are read: each such
statement stands directly behind a __syncwarp()."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_04579_gb300", "csrc")
# bar.sync is barrier.sync.aligned
ALIGNED = re.compile(r'asm volatile\(\s*"(bar\.sync|barrier\.sync\.aligned|barrier\.cluster\.[a-z.]*aligned|tcgen05\.ld\.)')


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_reconverged(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    for m in ALIGNED.finditer(text):
        before = text[: m.start()].rstrip()
        assert before.endswith("__syncwarp();"), text[m.start() : m.end() + 40]


def test_every_form_is_found():
    found = {m.group(1) for p in glob.glob(os.path.join(CSRC, "*.cu*")) for m in ALIGNED.finditer(open(p).read())}
    assert {"bar.sync", "tcgen05.ld."} <= found and any(f.startswith("barrier.cluster") for f in found)
