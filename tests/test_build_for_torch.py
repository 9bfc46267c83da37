"""The extension module uses torch's C++ interface: one built for another torch is neither taken for up to date nor loaded."""
import subprocess
import sys
from pathlib import Path

from paper_1909_05840_b200 import build as qb_build

ROOT = Path(__file__).resolve().parent.parent

OTHER_TORCH = """
import torch
torch.__version__ = "0.0.0+other"
import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import build
assert build.needs_build(), "an extension for another torch counts as built"
try:
    qb._ext()
except qb.QbertError as e:
    assert "paper_1909_05840_b200.build" in str(e)
else:
    raise AssertionError("an extension for another torch was loaded")
"""


def test_extension_of_another_torch_is_not_used():
    qb_build.build()
    assert not qb_build.needs_build()
    subprocess.run([sys.executable, "-c", OTHER_TORCH], check=True, cwd=ROOT)
