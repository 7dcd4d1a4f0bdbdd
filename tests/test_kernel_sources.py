"""Rules that every kernel source keeps and no GPU run can show."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_01464_gb300", "csrc")


def _code(path):
    """The source without its comments."""
    text = open(path).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name", sorted(os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cu*"))))
def test_no_multicast_loads(name):
    # the library also serves one process per GPU on several GPUs, where a load
    # into several CTAs' shared memory is not to be used
    for line in re.findall(r"cp\.async\.bulk[^;]*;", _code(os.path.join(CSRC, name))):
        assert "multicast" not in line, line
