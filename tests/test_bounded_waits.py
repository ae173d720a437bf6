"""No bounded wait of the digit-product kernels is ignored (no GPU): a wait that runs out leaves a copy or an MMA in
flight, so going on as if it had come uses memory that is still being written.  Only the drains that follow a set error
word may drop the result."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1611_06892_gb300", "csrc")
CALL = re.compile(r"\b(mbar_wait|wait_v)\s*\(")


def dropped(lines):
    """(line number, text) of wait calls whose result is not used: those that begin a statement."""
    out = []
    for i, line in enumerate(lines):
        code = line.split("//")[0]
        for m in CALL.finditer(code):
            before = code[:m.start()].rstrip()
            if before == "" or before[-1] in "{};" or re.search(r"(^|\s)(if|for|while)\s*\(.*\)$|\belse$", before):
                out.append((i, line.strip()))
    return out


@pytest.mark.parametrize("name", ["update_digits.cuh", "panel_digits.cuh"])
def test_results_of_bounded_waits_are_used(name):
    with open(os.path.join(CSRC, name)) as fh:
        lines = fh.read().split("\n")
    for i, text in dropped(lines):
        assert any("DERR_TIMEOUT" in x for x in lines[max(0, i - 3):i]), f"{name}:{i + 1}: {text}"
