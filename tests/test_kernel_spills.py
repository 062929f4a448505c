"""No mixed-precision kernel with output times and pathlines spills registers
(ptxas' report of the built library): at 64 registers they did, and lost 10 %."""
import os
import re
import subprocess

from paper_2302_13590_gb300 import _build


def test_mixed_kernels_with_times_and_paths_do_not_spill():
    log = os.path.join(_build.BUILD, "mp_mixed.o.log")
    _build.build_lib()
    if not os.path.exists(log):
        _build.build_lib(force=True)
    found = {}
    name = None
    for line in open(log):
        m = re.search(r"(?:Compiling entry function '|Function properties for )(\w+)", line)
        name = m.group(1) if m else name
        m = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", line)
        if m:
            found[name] = (int(m.group(1)), int(m.group(2)))
    names = subprocess.run(["c++filt"], input="\n".join(found), capture_output=True, text=True, check=True).stdout.split("\n")
    both = {n: v for n, v in zip(names, found.values()) if re.search(r"k_track_(static|dynamic)<.*, true, true>", n)}
    assert len(both) == 4, names
    assert all(v == (0, 0) for v in both.values()), both
