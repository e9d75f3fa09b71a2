"""The branch-free root, reciprocal and quotient equal the IEEE operations at the
ends of their stated range (tests/rounding_range.cu)."""
import os
import subprocess

import pytest

from .test_gpu_small import slpic  # noqa: F401

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_branch_free_operations_at_the_ends_of_their_range(slpic, tmp_path):  # noqa: F811
    from paper_2103_12194_gb300 import build
    exe = str(tmp_path / "rounding_range")
    subprocess.check_call([build.nvcc()] + build.common_flags() +
                          ["-I", build.CSRC, os.path.join(HERE, "rounding_range.cu"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
    assert out.stdout.split()[:5] == ["0", "0", "0", "of", str(1 << 32)], out.stdout
