"""A change to any file that the CUDA sources include makes the library out of date."""
import os
import re

from paper_2510_27258_gb300 import build


def test_every_included_file_is_a_build_input():
    known = {os.path.basename(f) for f in build.inputs()}
    for src in build.inputs():
        if not src.endswith(".py"):
            for name in re.findall(r'#include "([^"]+)"', open(src).read()):
                assert name in known, (src, name)
