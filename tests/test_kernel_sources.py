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
