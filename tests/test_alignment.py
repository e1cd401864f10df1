"""What the kernels copy or access 16 bytes at a time is declared with that
alignment, not left to where the toolchain places it: the noise tables (staged
by 16-byte asynchronous copies) and the rows' state in local memory."""
import shutil

import pytest


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not available")
def test_vector_accesses_are_to_aligned_objects():
    from tests import plan_probe
    tables, local_rows = plan_probe.alignments()
    assert tables >= 16 and local_rows >= 16
