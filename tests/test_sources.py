"""Rules of the kernel sources that no run would show."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_read_only_loads_in_kernels_that_start_early():
    """The kernels of an update may start while the one before them on the stream
    still writes; __ldg (ld.global.nc) is for memory that nobody writes while the
    kernel runs, so the layers and the caller's points are read with plain loads."""
    files = glob.glob(os.path.join(ROOT, "paper_2204_12876_gb300", "csrc", "*.cu*"))
    code = {f: re.sub(r"//[^\n]*", "", open(f).read()) for f in files}
    assert any("griddepcontrol.wait" in c for c in code.values())
    bad = [(os.path.basename(f), m) for f, c in code.items() for m in re.findall(r"__ldg\w*|ld\.global\S*\.nc", c)]
    assert not bad, bad
