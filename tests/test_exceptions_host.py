"""No C++ exception can leave the C entries for want of host memory on the way
through pic_create: the library's arrays come from malloc, from new with
nothrow, or are static."""
import subprocess

import __graft_entry__ as g
from paper_2602_15130_gb300 import _build


def test_no_throwing_array_new():
    g.build()
    names = subprocess.run(["nm", "-D", "--undefined-only", str(_build.LIB)], capture_output=True, text=True,
                           check=True).stdout
    assert "_Znam" not in {line.split()[-1].split("@")[0] for line in names.splitlines() if line.strip()}
