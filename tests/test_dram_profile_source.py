"""The source whose hash guards the DRAM figures of the bidirectional search holds the sizes it is built with."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2306_03651_gb300", "csrc")


def test_search_sizes_are_in_the_hashed_source():
    sizes = {f: re.findall(r"using Log\w+ = LogCfg<[^>]+>", open(os.path.join(CSRC, f)).read())
             for f in os.listdir(CSRC)}
    hashed = bench.DRAM_PROFILES["bidir"][1]
    assert len(sizes[hashed]) == 3 and not any(v for f, v in sizes.items() if f != hashed)
