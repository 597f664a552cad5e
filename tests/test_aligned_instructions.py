"""Instructions of the form .sync.aligned are undefined in a warp whose lanes have parted:
every helper that holds one rejoins the lanes first."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2510_00566_gb300", "csrc")
SOURCES = [f for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))]


def _aligned(line):
    return ".sync.aligned" in line


@pytest.mark.parametrize("name", [f for f in SOURCES
                                  if any(map(_aligned, open(os.path.join(CSRC, f))))])
def test_lanes_rejoin_before_an_aligned_instruction(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    # helpers that hold such an instruction: from the signature to the closing brace
    bodies = [m for m in re.finditer(r"\n__device__ __forceinline__ [^;{]*\{\n(.*?)\n\}(?=\n)", text, re.S)
              if _aligned(m.group(1))]
    assert sum(len(re.findall(r"\basm volatile\(", m.group(1))) for m in bodies) >= \
        sum(1 for line in text.split("\n") if _aligned(line)), "an aligned instruction outside a helper"
    for m in bodies:
        before = m.group(1).split(".sync.aligned")[0]
        assert "__syncwarp();" in before, m.group(0).split("{")[0]
