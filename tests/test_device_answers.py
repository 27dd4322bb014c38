"""What a kernel launcher asks the CUDA runtime about the device is kept per device (CPU: the sources are read): the library takes a
device per context, and an answer in a static belongs to whichever device was current at the first call."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_01662_b200", "csrc")
ASKS = r"cudaOccupancy\w+|cudaDeviceGetAttribute|cudaGetDeviceProperties|resident_clusters"


def test_no_answer_about_a_device_is_kept_in_a_static():
    asked = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh", ".h")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        asked += len(re.findall(ASKS, text))
        for m in re.finditer(r"\bstatic\b[^;{(]*(?:=|\{|\[)[^;]*;", text):   # a static with an initialiser
            assert not re.search(ASKS, m.group(0)), (name, m.group(0)[:120])
    assert asked >= 4
