"""The incremental build: what a change rebuilds."""
import os
import re

from paper_2601_04904_gb300 import build


def test_every_included_file_counts_as_a_header():
    """A change of any file that a translation unit includes rebuilds the units."""
    headers = {os.path.realpath(h) for h in build._headers()}
    for src in build._sources():
        for inc in re.findall(r'#include "([^"]+)"', open(src).read()):
            assert os.path.realpath(os.path.join(build.CSRC, inc)) in headers, (os.path.basename(src), inc)
