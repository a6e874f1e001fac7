"""Properties of the kernels' sources that no run on one GPU can show."""
import os
import re

from paper_2211_10725_gb300 import build_lib


def test_no_load_writes_another_blocks_shared_memory():
    """One library serves every rank of a multi-GPU run, so none of its bulk
    loads may be a cluster multicast (a completion signal to both blocks of a
    pair moves no data and is fine)."""
    src = os.path.join(build_lib.PKG, "csrc")
    loads = 0
    for name in sorted(os.listdir(src)):
        with open(os.path.join(src, name)) as f:
            for instr in re.findall(r"cp\.async\.bulk[\w.:]*", f.read()):
                loads += 1
                assert "multicast" not in instr, (name, instr)
    assert loads > 5
