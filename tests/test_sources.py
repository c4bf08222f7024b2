"""Rules that the CUDA sources keep, read as text."""

import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2210_11295_gb300" / "csrc"


def test_copies_stay_within_one_cta():
    """Replicas on several GPUs run the same kernels, so no bulk or tensor copy
    writes into another CTA's shared memory."""
    for path in sorted(CSRC.glob("*.cu*")):
        code = re.sub(r"//[^\n]*", "", path.read_text())
        assert ".multicast" not in code, path.name
