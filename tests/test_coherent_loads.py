"""Kernels are set up while the kernel before them on the stream still runs, so that nothing that kernel may have
written is read-only for their lifetime: no non-coherent load, and no argument that the compiler may read with one."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_1909_05840_b200" / "csrc"


def code(path: Path) -> str:
    return re.sub(r"//[^\n]*", "", path.read_text())


@pytest.mark.parametrize("path", sorted([*CSRC.glob("*.cu"), *CSRC.glob("*.cuh")]), ids=lambda p: p.name)
def test_no_read_only_loads(path):
    text = code(path)
    for pattern in (r"__ldg\s*\(", r"\bld\.global(\.\w+)*\.nc\b", r"\bconst\s+\w+\s*\*\s*(const\s+)?__restrict__"):
        found = re.search(pattern, text)
        assert found is None, f"{path.name}: {found.group(0)}"
