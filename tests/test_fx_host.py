"""The fixed-point arithmetic of the FP64-class passes (csrc/fx64.cuh), compiled for the host: register DFTs,
products and FP64 decoding against long double, at the bounds the passes reach."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_07777_gb300", "csrc")


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("fx") / "fx_check")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, os.path.join(ROOT, "tests", "host", "fx_check.cu"), "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([out], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
    return {ln.split()[0]: float(ln.split()[1]) for ln in r.stdout.splitlines()}


# each rounded product is off by at most half a unit plus the dropped low product (a quarter unit) per part,
# sqrt(2) for the pair: 1.1; a DFT output sums the errors of its rotated inputs (radix 16: three rotations in
# a chain of at most 9 terms; radix 9: two levels of three)
BOUND = {2: 0.1, 3: 1.6, 4: 0.1, 6: 3.2, 8: 3.2, 9: 8.0, 12: 6.4, 16: 10.0}


@pytest.mark.parametrize("R", sorted(BOUND))
def test_register_dfts_match_the_definition(errors, R):
    assert errors[f"dft{R}"] < BOUND[R]
    assert errors[f"dft{R}_inv"] < BOUND[R]


def test_products_and_decoding(errors):
    assert errors["cmul"] < 1.5      # two parts of at most 0.5 + 0.25 + 0.25 units
    assert errors["mul"] < 1.0
    assert errors["decode"] <= 0.5 and errors["decode_all"] <= 0.5   # rounded to nearest
    assert errors["decode_df"] <= 1.0   # two floats, half a unit each
    assert errors["zero"] == 0 and errors["subnormal"] == 0
    assert errors["shr_even"] == 207


def test_green_products_keep_their_own_exponent(errors):
    assert errors["green"] < 1.0     # half a unit and the dropped low product (a quarter), of each product's own unit
    assert errors["align"] <= 0.5    # one rounding at the scale of the lane's largest product


def test_decoding_has_no_preferred_direction(errors):
    """Mean error over 100000 positive values, uniform and at each distance below the lane's largest: truncation has half
    a unit, rounding to nearest a standard error of 0.3 / sqrt(100000) = 0.001 and the ties' bias, in all 2^-5 / 4 +
    2^-6 / 8 + ... = 0.0104 of a unit for uniform values."""
    assert errors["decode_mean"] < 0.015 and errors["decode_binade"] < 0.01
