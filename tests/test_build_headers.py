"""The build recompiles a translation unit when any header it may include is newer."""
import glob
import os

from paper_2507_23602_gb300 import _build


def test_every_header_counts():
    here = os.path.dirname(os.path.abspath(_build.__file__))
    local = {f for f in glob.glob(os.path.join(here, "csrc", "*")) if f.endswith((".h", ".cuh", ".hpp"))}
    assert any(f.endswith(".h") for f in local) and local <= set(_build._headers())
