"""Checks of internal entry points through small native programs linked with the library."""
import os
import shutil

import pytest

from native_build import run

needs_nvcc = pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                                reason="nvcc not available")


@needs_nvcc
def test_operand_without_planes_is_not_marked_prepared(tmp_path):
    [(code, nmod)] = run("operand_alloc_check", tmp_path)
    assert code != 0 and nmod == 0
