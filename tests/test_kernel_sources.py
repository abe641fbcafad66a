"""What the CUDA sources must not contain, read as text (no GPU)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1005_0542_gb300", "csrc")


def test_no_multicast_loads():
    # one library serves single-GPU programs and the replicas of a multi-GPU run: no bulk copy of it
    # writes into the shared memory of several CTAs of a cluster
    files = [f for ext in ("cu", "cuh", "h") for f in glob.glob(os.path.join(CSRC, "*." + ext))]
    assert len(files) > 10
    for f in files:
        for asm in re.findall(r"cp\.async\.bulk[a-z0-9_.:]*", open(f).read()):
            assert "multicast" not in asm, (os.path.basename(f), asm)
