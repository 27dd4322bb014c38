"""No experiment stays in the kernels behind a switch that no build sets (CPU: the sources are read)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_01662_b200", "csrc")
SWITCHES = {"LSA_CHECK",      # the checking build (build.py --check)
            "LSA_TIMELINE"}   # clock stamps of the fine kernel, for profiles


def test_conditional_code_belongs_to_a_build():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(CSRC, name)) as f:
                for line in re.findall(r"^[ \t]*#[ \t]*(?:if|ifdef|ifndef|elif)\b.*", f.read(), re.M):
                    assert set(re.findall(r"\bLSA_\w+", line)) <= SWITCHES, (name, line)
