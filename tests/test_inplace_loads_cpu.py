"""The time loop writes the next level over u^{n-1}, so no kernel may read u^{n-1}
through the read-only path (__ldg, or a __restrict__ pointer that lets the
compiler take it): CUDA asks that such memory stay unwritten while the kernel
runs.  The loads are plain C++ that no result shows; this reads the sources."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_1308_3214_gb300" / "csrc"


@pytest.mark.parametrize("name", sorted(p.name for p in CSRC.glob("*.cu*")))
def test_previous_level_is_read_by_plain_loads(name):
    text = (CSRC / name).read_text()
    for m in re.finditer(r"^.*\b(\w+)\s*=\s*[^;\n]*\bup_(?:hi|lo)\b[^;\n]*;", text, re.M):
        line, var = m.group(0), m.group(1)
        if "*" not in line.split("=")[0]:
            continue                                   # not a pointer of its own
        assert "__restrict__" not in line, line
        assert not re.search(r"__ldg\(\s*" + var + r"\b", text), line
    assert not re.search(r"__ldg\([^()]*\bup_(hi|lo)\b", text)


def test_float64_fields_are_read_by_plain_loads():
    """f64_each reads every field of a float64 pass, u^{n-1} among them."""
    text = (CSRC / "molt_f64.cuh").read_text()
    head = re.search(r"void f64_each\(([^)]*)\)", text).group(1)
    assert "__restrict__" not in head
