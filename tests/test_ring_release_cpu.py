"""Rings of shared-memory stages in the tensor-memory gradient kernels: the producer's wait for a stage, as the source has it, in a model of
mbarrier parities where the producer may be late by any number of tiles."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_08874_b200", "csrc")


def ring_of(name):
    """(stages, barriers that release them, tile -> barrier, tile -> awaited phase) of the producer's wait in a source file."""
    src = open(os.path.join(CSRC, name)).read()
    stages = int(re.search(r"\bkStages = (\d+)", src).group(1))
    m = re.search(r"if \(i >= (?:kStages|2)\) wait_spin\(pp, (BAR_\w+) \+ (.+?), (.+?), kTimeoutRole\);", src)
    bar, index, phase = m.groups()
    count = int(re.search(rf"\b{bar} = \d+;\s*// \[(\d)\]", src).group(1))

    def value(text, i):
        text = re.sub(r"\bkStages\b", str(stages), text).replace("/", "//")
        return eval(text, {"__builtins__": {}}, {"i": i, "b": i & 1, "s": i % stages})
    return stages, count, lambda i: value(index, i), lambda i: value(phase, i)


@pytest.mark.parametrize("name", ["bwd_values_umma.cu", "bwd_umma.cu", "bwd_terms_umma.cu"])
@pytest.mark.parametrize("late", [False, True], ids=["at_once", "late"])
def test_producer_is_never_overtaken(name, late):
    stages, count, barrier, phase = ring_of(name)
    done = [0] * count                                     # phases completed by the consumer, tile after tile
    consumed = 0
    for i in range(64):
        if i >= stages:
            b = barrier(i)
            # late: every tile that has been loaded is consumed before the producer looks
            while consumed < (i if late else i - stages + 1):
                done[consumed % count] += 1
                consumed += 1
            assert done[b] % 2 != phase(i) % 2, f"tile {i}: the wait for phase {phase(i)} of barrier {b} meets phase {done[b]}"
            assert done[b] > phase(i), f"tile {i}: its stage has not been released"
