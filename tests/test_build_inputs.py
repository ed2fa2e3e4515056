"""The library is built again when any file it is compiled from is newer."""

import os
import re

from paper_2606_14782_gb300 import build


def test_every_included_file_is_watched():
    watched = set(build.inputs())
    todo = [p for p in watched if p.endswith(".cu")]
    assert len(todo) >= 7
    seen = set()
    while todo:
        path = todo.pop()
        seen.add(path)
        assert path in watched, path
        with open(path) as f:
            names = re.findall(r'#include "([^"]+)"', f.read())
        for name in names:
            places = [os.path.join(d, name) for d in (build.CSRC, os.path.join(build.ROOT, "include"))]
            found = [p for p in places if os.path.exists(p)]
            assert found, (path, name)
            todo += [p for p in found if p not in seen]
