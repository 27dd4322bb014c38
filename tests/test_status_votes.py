"""The kernels' decision to give up is one per block (CPU: the sources are read).  A thread that looks at the status word for itself may
see it raised where its neighbour does not; one of them then waits for ever on a barrier that counts both."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_01662_b200", "csrc")


def _sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, name)) as f:
                yield name, f.read()


def test_a_block_gives_up_by_a_vote():
    votes = 0
    for name, text in _sources():
        if name == "lsa_tc.cuh":
            assert "return __syncthreads_or(status_raised(status)) != 0;" in text
            continue
        votes += len(re.findall(r"block_gives_up\(p\.status\)", text))
        for m in re.finditer(r"[^\n]*status_raised\([^\n]*", text):
            # a thread's own look goes nowhere but into a vote of its block
            own = re.fullmatch(r"\s*const bool (\w+) = tc::status_raised\(p\.status\);.*", m.group(0))
            assert own, (name, m.group(0))
            uses = re.findall(rf"\b{own.group(1)}\b", re.sub(r"//[^\n]*", "", text[m.end():]))
            assert uses == [own.group(1)] and f"__syncthreads_or({own.group(1)})" in text, (name, own.group(1))
    assert votes >= 6


def test_waits_before_a_counted_barrier_are_voted_on():
    """Where a named barrier counts the threads of several warps, the outcome of a wait before it is agreed on."""
    for name, text in _sources():
        if "bar.sync %0, %1" in text and "mbar_wait" in text:
            assert "tc::all_of<" in text, name
