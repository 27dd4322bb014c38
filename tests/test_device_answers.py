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


def test_no_rule_names_the_sms_of_one_chip():
    """148 stands only where a call has no device's count to go by."""
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(CSRC, name)) as f:
                code = re.sub(r"//[^\n]*", "", f.read())
            for line in code.split("\n"):
                assert not re.search(r"\b(148|1184|296)\b", line) or re.search(r"\? [\w.]+ : 148\b|return 148;|n = 148;", line), (name, line)
