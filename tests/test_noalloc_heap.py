"""The allocation-free step uses no heap on the host either: the translation units
it runs through (its own and the FP64 kernels' host code, which lays the network
out) refer to no allocation function."""
import os
import shutil
import subprocess

import pytest


@pytest.mark.parametrize("unit", ["noalloc", "fp64"])
def test_no_heap_in_the_allocation_free_step(unit):
    from paper_2207_08500_gb300 import build
    if shutil.which("nm") is None:
        pytest.skip("needs nm")
    build.build()
    out = subprocess.run(["nm", "-u", os.path.join(build.BUILD, unit + ".o")], capture_output=True, text=True,
                         check=True).stdout
    names = [line.split()[-1] for line in out.splitlines() if line.strip()]
    assert names
    # operator new and new[] of any form, and the C functions
    assert not [n for n in names if n.startswith(("_Znw", "_Zna")) or n in ("malloc", "calloc", "realloc")]
