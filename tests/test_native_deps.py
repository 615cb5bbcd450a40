"""Every file that a translation unit includes makes the library stale (CPU)."""
import os
import re

from paper_2601_01903_gb300 import native


def test_included_files_are_dependencies():
    known = {os.path.realpath(p) for p in native._deps()}
    for src in list(known):
        with open(src) as f:
            for name in re.findall(r'^\s*#include "([^"]+)"', f.read(), flags=re.M):
                found = [os.path.join(d, name) for d in (os.path.dirname(src), native.INCLUDE)]
                here = [os.path.realpath(p) for p in found if os.path.exists(p)]
                assert here and here[0] in known, (src, name)
