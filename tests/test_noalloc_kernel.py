"""The allocation-free sampler runs the search's instantiation without the ob, RTB
and fsfm parts (with them its calls took up to twice as long): what the library
built here contains and what the sampler's object refers to (no GPU needed)."""
import os
import shutil
import subprocess

import pytest


def test_sampler_has_its_own_instantiation():
    from paper_2304_08356_gb300 import build as B
    if shutil.which("nm") is None:
        pytest.skip("nm not available")
    B.build()
    names = subprocess.run(["nm", os.path.join(B.BUILD, "k_bfs.o")], capture_output=True, text=True, check=True).stdout
    assert "k_bfsILb0ELi512ELb0EE" in names            # k_bfs<false, 512, false>
    refs = subprocess.run(["nm", "-u", os.path.join(B.BUILD, "api_noalloc.o")], capture_output=True, text=True,
                          check=True).stdout
    assert "launch_bfs_sampler" in refs
