"""The library is rebuilt when any file that its sources include changes."""
import os
import re

from paper_2003_13493_gb300 import build


def test_every_included_file_is_watched():
    watched = {os.path.realpath(p) for p in build._deps()}
    todo, seen = list(build._sources()), set()
    while todo:
        path = os.path.realpath(todo.pop())
        if path in seen:
            continue
        seen.add(path)
        with open(path) as f:
            for name in re.findall(r'#include "([^"]+)"', f.read()):
                here = os.path.join(os.path.dirname(path), name)
                todo.append(here if os.path.exists(here) else os.path.join(build.INCLUDE, name))
    assert seen <= watched, sorted(seen - watched)
