"""What the device sources must not contain, checked on their text (no GPU)."""
import glob
import os

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1304_5583_gb300", "csrc")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_a_cta_loads_into_its_own_shared_memory_only(path):
    """One library serves every process of a run on several GPUs, where copies
    that the memory system fans out to several CTAs are not used."""
    with open(path, encoding="utf-8") as f:
        assert "multi" + "cast" not in f.read()
