"""What short_select asks of its callers (CPU: the sources are read): it reads its keys 16 bytes at a time."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_01662_b200", "csrc")


def test_key_arrays_are_declared_aligned():
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        if "short_select<" not in text:
            continue
        arrays = re.findall(r"^(.*)\buint32_t keys\[kMaxSlots\w*\];", text, re.M)
        assert arrays, name
        for before in arrays:
            assert "alignas(16)" in before, (name, before)
        seen += len(arrays)
    assert seen == 5
