"""What the build counts as a reason to compile again."""
import os
import re

from paper_2105_07298_gb300 import build as apsp_build


def test_every_included_header_is_a_dependency():
    deps = {os.path.realpath(d) for d in apsp_build._deps()}
    for f in sorted(os.listdir(apsp_build.CSRC)):
        src = open(os.path.join(apsp_build.CSRC, f)).read()
        for h in re.findall(r'^#include "([^"]+)"', src, flags=re.M):
            assert os.path.realpath(os.path.join(apsp_build.CSRC, h)) in deps, (f, h)
