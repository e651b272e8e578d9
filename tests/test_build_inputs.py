"""The build watches every file that its translation units include."""
import os
import re

from paper_1705_10218_gb300 import build


def test_every_included_file_is_watched():
    watched = {os.path.realpath(p) for p in build.sources() + build.headers()}
    included = set()
    for path in watched:
        with open(path) as f:
            names = re.findall(r'^#include "([^"]+)"', f.read(), re.M)
        for name in names:
            found = [p for d in (build.CSRC, os.path.join(build.ROOT, "include"))
                     if os.path.exists(p := os.path.join(d, name))]
            assert found, name
            included.add(os.path.realpath(found[0]))
    assert included and included <= watched
