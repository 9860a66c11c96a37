"""Every header that a source file includes is one that build() watches: an
object is compiled again when any of them changes.  No GPU."""
import os
import re

from paper_2509_16407_gb300 import build as b


def test_included_headers_are_watched():
    watched = {os.path.realpath(h) for h in b._headers()}
    todo, seen = [os.path.realpath(s) for s in b._sources()], set()
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        for inc in re.findall(r'^\s*#\s*include\s+"([^"]+)"', open(f).read(), re.M):
            for d in (os.path.dirname(f), b.INCLUDE):  # the order in which the compiler looks
                h = os.path.realpath(os.path.join(d, inc))
                if os.path.exists(h):
                    assert h in watched, (f, inc)
                    todo.append(h)
                    break
            else:
                raise AssertionError(f"{f} includes {inc}, which is nowhere")
    # one copy of the public header
    names = [os.path.basename(h) for h in watched]
    assert len(names) == len(set(names)), sorted(names)
