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


@needs_nvcc
def test_two_pass_fft_code_on_host_at_every_compiled_length(tmp_path):
    rows = run("fft_lengths_check", tmp_path)
    assert [int(r[0]) for r in rows] == [16, 20, 24, 30, 32, 36, 40, 45, 48, 54, 60, 64, 72, 80, 90, 96, 100, 108]
    for n, f64, g64, f32, g32 in rows:  # the tolerances of the check at the other lengths
        assert f64 < 2e-15 and g64 < 2e-15, n
        assert f32 < 1e-6 and g32 < 1e-6, n


@pytest.mark.gpu
def test_lower_product_with_split_keeps_the_upper_triangle(tmp_path):
    rows = run("lower_split_check", tmp_path)
    assert len(rows) == 8
    for size, n, k, changed, err in rows:
        assert changed == 0, (size, n, k)
        # 2 k + 8 roundings of terms of magnitude one
        assert err <= (2 * k + 8) * (2.0 ** -53 if size == 8 else 2.0 ** -24), (size, n, k)


@pytest.mark.gpu
def test_double_float_conversions_round_as_the_fp64_unit(tmp_path):
    [(n, nv, bad, badv)] = run("df_store_check", tmp_path)
    assert n > 100000 and nv > 100000
    assert bad == 0 and badv == 0


@pytest.mark.gpu
def test_cholesky_and_triangular_solve_round_once_per_operation(tmp_path):
    [(nq, bad, nt, badt)] = run("quotient_check", tmp_path)
    assert nq > 15000 and nt > 400000
    # a product of relative size 2^-24 moves a rounding in about one of 2^20 values, the
    # reciprocals' own errors in fewer
    assert bad <= 1e-4 * nq and badt <= 1e-4 * nt
