"""What the kernels' sources must not hold."""

import os
import re

import paper_2104_09857_gb300

CSRC = os.path.join(os.path.dirname(paper_2104_09857_gb300.__file__), "csrc")


def test_no_multicast_loads():
    """The library serves one rank per GPU in multi-rank runs: every tile is
    loaded by the CTA that uses it, none is multicast to a cluster."""
    found = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".h")):
            with open(os.path.join(CSRC, name)) as f:
                found += [f"{name}:{i}" for i, line in enumerate(f, 1) if re.search(r"multicast", line)]
    assert not found, found


def test_warps_wait_together():
    """What follows a wait of a whole warp are warp-wide instructions, so its
    result has to be one for all lanes (mbar_wait_warp): a lane that gives up
    alone would leave the others in them.  The plain wait is for the producer,
    which is one thread: warp 0's branch, and Sched::produce."""
    for name in ("k_emu.cu", "k_tc.cu"):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        text = re.sub(r"__device__ int produce\(.*?\n  }\n", "", text, flags=re.S)
        parts = re.split(r"\n  (?:} else )?if \(warp == [01]\) {\n(?=    (?:if \(lane == 0\)|//))", text)
        assert len(parts) == 3, name  # before warp 0's branch, it, and what follows
        for outside in (parts[0], parts[2]):
            assert not re.search(r"\bmbar_wait\(", outside), name
        assert re.search(r"\bmbar_wait\(", parts[1]), name
