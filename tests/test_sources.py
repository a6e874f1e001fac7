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


def test_pair_kernel_waits_for_every_arrival_from_the_other_block():
    """A commit of the pair kernel arrives in both blocks' shared memory at
    some later time; neither block may leave before its last ones are in.  A
    missing wait would show as a rare fault, so it is read from the source."""
    with open(os.path.join(build_lib.PKG, "csrc", "gemm_tcgen05.cu")) as f:
        text = f.read()
    kernel = text[text.index("gemm_pair_tcgen05(const"):]
    kernel = kernel[:kernel.index("tmem_dealloc_pair")]
    assert set(re.findall(r"tc_commit_pair\(&(\w+)\[", kernel)) == {"empty", "acc_full"}
    producer, rest = kernel.split("} else if (warp == 1) {", 1)
    # both blocks' producers, after their last issue, take the last use of every stage
    tail = producer[producer.rindex("tma_load_2d_pair("):]
    waits = [line for line in tail.splitlines() if "mbar_wait_bounded(&empty[" in line]
    assert len(waits) == 1 and "kDrainWaitNs" in waits[0]
    before = tail[:tail.index("mbar_wait_bounded(&empty[")]
    assert "j < n_issued" in before.splitlines()[-2] and "rank" not in before.splitlines()[-2]
    # and both blocks' epilogues every accumulator
    epilogue = rest[rest.index("} else {"):]
    assert "warp_wait_uniform(&acc_full[b]" in epilogue
