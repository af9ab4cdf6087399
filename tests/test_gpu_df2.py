"""The two-lane double-float operations (csrc/df2.cuh, packed FP32 instructions) against the
scalar ones (csrc/df.cuh), bit for bit, lane by lane, on a million pseudo-random lane pairs:
the operations of the direction and adjoint passes, the WENO5 offset of the direction pass (with
and without rescaling) and its squared smoothness indicators.  What has no scalar form in df.cuh
(df2_div, df2_div_ru, df2_rcp_ru, the offset) is written out in tests/cuda/df2_check.cu.  Then the
errors of the divisions, square roots and FP64 reciprocals.
The check is built here from its own source into a temporary library; nothing of it is in
libns3d.so."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
NAMES = ["add_fast", "sub", "mul_u", "mul", "sqr_u", "mul_f_u", "add_pos_u", "add_ordered_u", "add_ordered",
         "twice", "two_prod", "div", "weno_offset", "indicator_B1", "indicator_B2", "indicator_B3",
         "weno_offset_rescaled", "div_ru", "rcp_ru"]
# relative errors in units of u^2 = 2^-48 (u = 2^-24): first-order bounds, and the means that the comments state.
# A division's remainder, of up to 4 u (seed error 2 u unrefined: 5 u), rounds three times on the way to it
# (2 + 3 + 4, 3 + 4 + 5) and is multiplied by a reciprocal in error by the seed's u (2 u), y.lo and a rounding:
# 9 + 4 * 3 (12 + 5 * 4), and a rounding of the result; 3 + 2 * 3 for a reciprocal (no x.lo).  A root's
# correction: half of the remainder's roundings 4 + 5, 2.5 u times the error of its factor (4 u, refined 3 u),
# and unrefined the second-order term (2.5 u)^2 / 2
ERRORS = {"df_div": (33, 0.66), "df2_div": (33, 0.63), "df_div_r": (22, 0.60), "df2_div_ru": (22, 0.60),
          "df2_rcp_ru": (9.5, 0.40), "df_sqrt": (18.5, 0.33), "df_sqrt_r": (13, 0.31)}


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2211_16718_gb300 import build as B
    out = str(tmp_path_factory.mktemp("df2") / "libdf2check.so")
    cmd = [B.nvcc()] + B.ARCH + ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", B.INCLUDE, "-I",
                                 B.CSRC, os.path.join(HERE, "cuda", "df2_check.cu"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(out)
    lib.df2_check.restype = ctypes.c_int
    lib.df2_check.argtypes = [ctypes.c_int, ctypes.c_ulonglong, ctypes.POINTER(ctypes.c_int)]
    lib.df2_check_nops.restype = ctypes.c_int
    assert lib.df2_check_nops() == len(NAMES)
    lib.error_check.argtypes = [ctypes.c_int, ctypes.c_ulonglong, ctypes.c_void_p, ctypes.c_void_p]
    assert lib.error_check_nops() == len(ERRORS)
    return lib


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [1, 20261204])
def test_two_lane_double_float_equals_scalar_bitwise(checker, seed):
    bad = (ctypes.c_int * len(NAMES))()
    assert checker.df2_check(1 << 20, seed, bad) == 0
    mismatches = {n: bad[i] for i, n in enumerate(NAMES) if bad[i]}
    assert not mismatches, mismatches


# bounds: the final rounding (0.5 ulp) and the seed's error cubed (it is below 2^-18, so 0.13 ulp at
# most), and for the root half of the rounding of x r (0.5 ulp)
@pytest.mark.gpu
@pytest.mark.parametrize("what,bound", [(0, 0.6), (1, 1.1)])
def test_cubic_reciprocals_of_the_all_fp64_mode(checker, what, bound):
    """rcp_cubic and rsqrt_cubic (csrc/k_dir_impl.cuh) over every exponent: the error in ulps, and
    the IEEE results for zero, subnormal, overflowing and infinite operands and for NaN."""
    ulp, bad = ctypes.c_int(), ctypes.c_int()
    for seed in (1, 20261205):
        assert checker.cubic_check(what, ctypes.c_ulonglong(seed), ctypes.byref(ulp), ctypes.byref(bad)) == 0
        assert bad.value == 0
        assert ulp.value * 1e-6 <= bound


@pytest.mark.gpu
def test_double_float_division_and_root_errors(checker):
    """Errors of the divisions and square roots on four million normalised operands."""
    mx, mean = (ctypes.c_double * len(ERRORS))(), (ctypes.c_double * len(ERRORS))()
    assert checker.error_check(1 << 22, 20261205, mx, mean) == 0
    for k, (name, (bound, avg)) in enumerate(ERRORS.items()):
        assert mx[k] <= bound and mean[k] <= avg, (name, mx[k], mean[k])
