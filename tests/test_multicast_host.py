"""The library runs as one replica per GPU in jobs of several, so no load of it is a
multicast into a cluster's shared memory."""
import glob
import os
import re

import paper_1512_06473_gb300.build as build


def test_no_multicast_loads():
    found = []
    for path in glob.glob(os.path.join(build.CSRC, "*.cu*")):
        text = open(path).read()
        text = re.sub(r"/\*.*?\*/|//[^\n]*", "", text, flags=re.S)
        for asm in re.findall(r'(?:"[^"\n]*"\s*)+', text):
            if "cp.async.bulk" in asm and "multicast" in asm:
                found.append((os.path.basename(path), asm))
    assert not found, found
