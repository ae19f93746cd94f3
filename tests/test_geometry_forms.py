"""CPU index checks of the step kernels' further forms (tests/geometry_forms_check.cu): band-limited
transforms, cut twiddle tables, in-place and lean bodies, the corrector's row kinds."""
import os
import re
import subprocess

import pytest

from test_geometry import ROOT, _nvcc

CSRC = os.path.join(ROOT, "paper_2304_03306_gb300", "csrc")


def test_every_form_stays_in_bounds(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc is not available")
    exe = str(tmp_path / "geometry_forms_check")
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC,
                        os.path.join(ROOT, "tests", "geometry_forms_check.cu"), "-o", exe],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-4000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-4000:]
    last = r.stdout.strip().splitlines()[-1]
    assert int(last.split()[0]) > 400 and last.endswith(" 0 failures"), last


def test_checker_covers_what_the_launchers_instantiate():
    impl = open(os.path.join(CSRC, "ttsh_ops_impl.cuh")).read()
    chk = open(os.path.join(ROOT, "tests", "geometry_forms_check.cu")).read()
    kinds = set(re.findall(r"launch_row_(?:kind|io)<T, N, (ROW_\w+)>", impl)) - {"ROW_STEP"}
    modes = set(re.findall(r"launch_col_mode<T, N, (COL_\w+)>", impl)) - {"COL_STEP"}
    assert {"ROW_FEATURES", "ROW_FWD_CORR"} <= kinds and "COL_PROLOGUE" in modes
    for k in kinds:
        assert f"check_row_form<T, N, {k}, R, RPE>()" in chk, k
    for m in modes:
        assert f"check_col_form<T, N, {m}, CPE>()" in chk, m
    # the shapes the checker takes for them are the launchers'
    assert "template <typename T, int N, int MODE, int PE = default_step_col_pe<T, N>()>\nstatic cudaError_t launch_col_mode" in impl
    assert "constexpr int R = default_rows<T, N>(), PE = default_row_pe<T, N>();\n  using Geo = RowGeo<T, N, KIND, R, PE>;" in impl
    # every step shape of the registry, in the form the launcher picks
    for pe in re.findall(r"add_col_variant<T, N, (\d+)>\(o\)", impl):
        assert f"check_col_step<T, N, {pe}>()" in chk, pe
    for rows, pe, rest in re.findall(r"add_row_variant<T, N, (\d+), (\d+)((?:, \d+)*)>\(o\)", impl):
        assert f"check_row_form<T, N, ROW_STEP, {rows}, {pe}{rest}>()" in chk, (rows, pe, rest)
